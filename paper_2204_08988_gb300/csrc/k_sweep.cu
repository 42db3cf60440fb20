// k_sweep.cu -- the label step and the sufficient statistics (Sec. 4.1 steps (e),
// (f); Sec. 4.4 "updating the sufficient statistics" in three steps).
//
//   labels       : z_i = argmax_k [log pi_k + log f(x_i; theta_k) + G_ik] on CUDA cores.
//                  labels_small: Gaussian, d <= 8 (FP64) or 16 (FP32), all clusters'
//                  parameters in shared memory.  labels_niw64: Gaussian FP64, scores
//                  enclosed in FP32 first.  labels_simt: what is left (FP32 at larger d or
//                  K_max, multinomial data, every score for the score hook), one thread
//                  per point, parameters staged in chunks and read by broadcast.
//   hist/scan/scatter : stable counting sort of the points by cluster (tiles of
//                  SORT_TILE points), so that the next kernel sees each cluster as one run.
//   substats     : per sorted run, z-bar_i from the two sub-clusters of z_i, then the
//                  per-sub-cluster sums of xt xt^T (xt = [x - shift_k, 1]) as 4x4
//                  register blocks, one partial record per (CTA, cluster) run.
//   combine      : sums each cluster's records in CTA order (deterministic).
#include <math.h>

#include <cuda_bf16.h>

#include <algorithm>

#include "dpmm_internal.cuh"

namespace dpmm {

template <typename T, typename XT>
__device__ inline T ldx(const XT* p) { return (T)(*p); }
template <>
__device__ inline float ldx<float, __nv_bfloat16>(const __nv_bfloat16* p) { return __bfloat162float(*p); }

__device__ __forceinline__ void mw_cp16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

template <typename T>
struct ParamView {
    const T* W;      // slots x d x d
    const T* mu;     // slots x d
    const T* c;      // slots
    const T* lt;     // slots x d (multinomial)
};

template <typename T>
__device__ inline T gumbel_of(uint32_t w0, uint32_t w1);
template <>
__device__ inline double gumbel_of<double>(uint32_t a, uint32_t b) {
    return -log(-log(u01_f64(a, b)));
}
template <>
__device__ inline float gumbel_of<float>(uint32_t a, uint32_t) {
    // the inner log must be accurate near u = 1 (-log u is as small as 6e-8 there)
    return -__logf(-logf(u01_f32(a)));
}
template <typename T>
__device__ inline T gmax();
template <>
__device__ inline double gmax<double>() { return GUMBEL_MAX_F64; }
template <>
__device__ inline float gmax<float>() { return GUMBEL_MAX_F32; }

// ------------------------------------------------------------------ labels (simt)
// Dynamic shared memory: CB clusters x (d*d + d + 1) T (d + 1 for multinomial), then
// blockDim x (d + 1) T point rows.
template <typename T, typename XT, bool SCORES>
__global__ void __launch_bounds__(256) labels_simt_kernel(int kind, int d, int xs, int64_t N, const XT* __restrict__ X,
                                                          ParamView<T> pv, const int* dK, const uint32_t* diter,
                                                          uint64_t seed, int CB, const int* gate,
                                                          double* scores, int32_t* z) {
    if (gate && *gate == 0) return;
    extern __shared__ __align__(16) unsigned char smraw[];
    T* sW = (T*)smraw;
    const int per = kind == DPMM_PRIOR_NIW ? d * d + d + 1 : d + 1;
    T* sx = sW + (size_t)CB * per;
    const int K = *dK;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int64_t ntiles = (N + nt - 1) / nt;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {  // grid-stride over point tiles
    __syncthreads();
    const int64_t i = tile * nt + tid;
    const bool live = i < N;
    T* xr = sx + (size_t)tid * (d + 1);
    if (live)
        for (int j = 0; j < d; ++j) xr[j] = ldx<T, XT>(X + i * xs + j);
    Key key{seed, diter[0], diter[1], diter[2]};
    T best = -INFINITY;
    int zb = 0;
    uint32_t w[4];
    int wblk = -1;
    for (int k0 = 0; k0 < K; k0 += CB) {
        const int nc = min(CB, K - k0);
        __syncthreads();
        for (int e = tid; e < nc * per; e += nt) {
            int cc = e / per, r = e % per;
            int s = 3 * (k0 + cc);
            T v;
            if (kind == DPMM_PRIOR_NIW) {
                if (r < d * d) v = pv.W[(size_t)s * d * d + r];
                else if (r < d * d + d) v = pv.mu[(size_t)s * d + (r - d * d)];
                else v = pv.c[s];
            } else {
                v = (r < d) ? pv.lt[(size_t)s * d + r] : pv.c[s];
            }
            sW[e] = v;
        }
        __syncthreads();
        if (!live) continue;
        for (int cc = 0; cc < nc; ++cc) {
            const T* Wk = sW + (size_t)cc * per;
            T sc;
            if (kind == DPMM_PRIOR_NIW) {
                const T* mk = Wk + d * d;
                T q = 0;
                for (int j = 0; j < d; ++j) {
                    T y = 0;
                    for (int l = 0; l <= j; ++l) y += Wk[l * d + j] * (xr[l] - mk[l]);
                    q += y * y;
                }
                sc = Wk[d * d + d] - (T)0.5 * q;
            } else {
                T a = 0;
                for (int j = 0; j < d; ++j) a += xr[j] * Wk[j];
                sc = Wk[d] + a;
            }
            const int k = k0 + cc;
            if constexpr (SCORES) scores[i * K + k] = (double)sc;
            if (sc + gmax<T>() > best) {  // otherwise k cannot win the argmax
                if ((k >> 1) != wblk) {
                    key.block((uint32_t)i, TAG_Z, (uint32_t)(k >> 1), w);
                    wblk = k >> 1;
                }
                T g = (k & 1) ? gumbel_of<T>(w[2], w[3]) : gumbel_of<T>(w[0], w[1]);
                T v = sc + g;
                if (v > best) {
                    best = v;
                    zb = k;
                }
            }
        }
    }
    if (live) z[i] = zb;
    }
}

// An FP64 Gumbel value to within GUMBEL_APPROX, in FP32 arithmetic: e = -log u from u, or
// from 1 - u (exact in the 53-bit integer) when u is above 1/2, to a few FP32 roundings, so
// log e is off by about 4e-7 and, for |log e| <= 37, its own rounding by 4e-6.
constexpr double GUMBEL_APPROX = 1e-4;
__device__ inline float gumbel_approx(uint32_t a, uint32_t b) {
    const unsigned long long m = 2ull * (((unsigned long long)(a >> 6) << 26) | (b >> 6)) + 1ull;
    const float s = 1.1102230246251565e-16f;  // 2^-53
    const float e = m < (1ull << 52) ? -logf((float)m * s) : -log1pf(-(float)((1ull << 53) - m) * s);
    return -logf(e);
}

// Two values s + G cannot be told apart by approximate G when they are this close: G's errors, and the
// rounding of the sums (size: their magnitude), which makes equals of them where s is large.
__device__ inline double approx_margin(double size) { return 4 * GUMBEL_APPROX + 1e-15 * size; }

template <typename T>
__device__ inline T gmin();  // below every Gumbel value of the precision
template <>
__device__ inline double gmin<double>() { return -3.7; }
template <>
__device__ inline float gmin<float>() { return -3.f; }

// ------------------------------------------------------------------ Gaussian labels, small d
// z_i = argmax_k [s_ik + G_ik] for d <= 16 (FP32) or d <= 8 (FP64).  The sums are short there,
// and what bounds the step is the chain of latencies of one point's K clusters; so L lanes share
// a point (clusters sub, sub + L, ...), as many as the points leave room for.  All clusters'
// parameters are staged in shared memory once per block, rows and columns padded with zeros
// to DV (a zero adds nothing to a sum).  A first pass finds the two best scores: if the second
// cannot win whatever the Gumbel values (monotone rounding makes the bounds hold for the
// rounded sums), the label is known.  Otherwise the clusters within reach of the best score
// are drawn; in FP64 by an FP32 value first (gumbel_approx), FP64 logarithms being taken for
// those it cannot tell apart.
// Measured: FP64, d = 2, K = 10, N = 10,000: 27 us, from 62 us with one thread per point
// and FP64 draws; FP32, d = 8, K = 12, N = 100,003: 25 us, from 35 us.
template <typename T, int DV, int L>
__global__ void __launch_bounds__(256) labels_small_kernel(int d, int xs, int64_t N, const T* __restrict__ X,
                                                           ParamView<T> pv, const int* dK, const uint32_t* diter,
                                                           uint64_t seed, int32_t* z) {
    extern __shared__ __align__(16) unsigned char smraw[];
    constexpr int PER = DV * DV + DV + 1;  // W, mu, c; odd: lanes of different clusters use different banks
    T* sp = (T*)smraw;
    const int K = *dK, tid = threadIdx.x, sub = tid % L;
    for (int e = tid; e < K * PER; e += 256) {
        const int k = e / PER, r = e % PER;
        const size_t s = 3 * (size_t)k;
        T v = 0;
        if (r < DV * DV) {
            const int l = r / DV, j = r % DV;
            if (l <= j && j < d) v = pv.W[s * d * d + l * d + j];
        } else if (r < DV * DV + DV) {
            if (r - DV * DV < d) v = pv.mu[s * d + (r - DV * DV)];
        } else {
            v = pv.c[s];
        }
        sp[e] = v;
    }
    __syncthreads();
    const Key key{seed, diter[0], diter[1], diter[2]};
    const int64_t step = (int64_t)gridDim.x * (256 / L);
    for (int64_t i0 = (int64_t)blockIdx.x * (256 / L) + (tid & ~31) / L; i0 < N; i0 += step) {  // uniform in a warp
        const int64_t ir = i0 + (tid & 31) / L;
        const bool live = ir < N;
        const int64_t i = live ? ir : N - 1;
        T x[DV];
#pragma unroll
        for (int j = 0; j < DV; ++j) x[j] = j < d ? X[i * xs + j] : (T)0;
        auto score = [&](int k) -> T {
            const T* P = sp + k * PER;
            T q = 0;
            T t[DV];
#pragma unroll
            for (int j = 0; j < DV; ++j) t[j] = x[j] - P[DV * DV + j];
#pragma unroll
            for (int j = 0; j < DV; ++j) {
                T y = 0;
#pragma unroll
                for (int l = 0; l <= j; ++l) y = fma(P[l * DV + j], t[l], y);
                q = fma(y, y, q);
            }
            return P[PER - 1] - (T)0.5 * q;
        };
        T best = -INFINITY, second = -INFINITY;
        int kb = 0;
        for (int k = sub; k < K; k += L) {
            const T s = score(k);
            if (s > best) {
                second = best;
                best = s;
                kb = k;
            } else if (s > second) {
                second = s;
            }
        }
#pragma unroll
        for (int o = 1; o < L; o <<= 1) {
            const T ob = __shfl_xor_sync(0xffffffffu, best, o), os = __shfl_xor_sync(0xffffffffu, second, o);
            const int ok = __shfl_xor_sync(0xffffffffu, kb, o);
            second = max(min(best, ob), max(second, os));
            if (ob > best || (ob == best && ok < kb)) {
                best = ob;
                kb = ok;
            }
        }
        const T reach = best + gmin<T>();
        const bool need = second > -INFINITY && !(second + gmax<T>() < reach);
        if (__any_sync(0xffffffffu, need)) {
            T vb = -INFINITY, vs = -INFINITY;  // the best value and the runner-up
            int kv = 0;
            uint32_t w[4];
            auto words = [&](int k) { key.block((uint32_t)i, TAG_Z, (uint32_t)(k >> 1), w); };
            if (need)
                for (int k = sub; k < K; k += L) {
                    const T s = score(k);
                    if (!(s > -INFINITY) || s + gmax<T>() < reach) continue;
                    words(k);
                    T v;
                    if constexpr (sizeof(T) == 8) v = s + (T)((k & 1) ? gumbel_approx(w[2], w[3]) : gumbel_approx(w[0], w[1]));
                    else v = s + ((k & 1) ? gumbel_of<T>(w[2], w[3]) : gumbel_of<T>(w[0], w[1]));
                    if (v > vb) {
                        vs = vb;
                        vb = v;
                        kv = k;
                    } else if (v > vs) {
                        vs = v;
                    }
                }
            auto reduce = [&]() {
#pragma unroll
                for (int o = 1; o < L; o <<= 1) {
                    const T ob = __shfl_xor_sync(0xffffffffu, vb, o), os = __shfl_xor_sync(0xffffffffu, vs, o);
                    const int ok = __shfl_xor_sync(0xffffffffu, kv, o);
                    vs = max(min(vb, ob), max(vs, os));
                    if (ob > vb || (ob == vb && ok < kv)) {
                        vb = ob;
                        kv = ok;
                    }
                }
            };
            reduce();
            if constexpr (sizeof(T) == 8) {
                const T cut = vb - approx_margin(fabs(vb));
                const bool near = need && vs >= cut;
                if (__any_sync(0xffffffffu, near)) {
                    const int keep = kv;
                    vb = vs = -INFINITY;
                    if (near)
                        for (int k = sub; k < K; k += L) {
                            const T s = score(k);
                            if (!(s > -INFINITY) || s + gmax<T>() < reach) continue;
                            words(k);
                            if (s + (T)((k & 1) ? gumbel_approx(w[2], w[3]) : gumbel_approx(w[0], w[1])) < cut) continue;
                            const T v = s + ((k & 1) ? gumbel_of<T>(w[2], w[3]) : gumbel_of<T>(w[0], w[1]));
                            if (v > vb) {
                                vb = v;
                                kv = k;
                            }
                        }
                    reduce();
                    if (!near) kv = keep;
                }
            }
            if (need) kb = kv;
        }
        if (live && sub == 0) z[i] = kb;
    }
}

// ------------------------------------------------------------------ Gaussian labels in FP64
// z_i = argmax_k [s_ik + G_ik], s_ik = c_k - 1/2 ||W_k^T (x_i - mu_k)||^2, one thread per
// point.  What bounds the step is the FP64 pipe (two lanes an SM): scoring every cluster
// takes K d^2 / 2 FP64 multiply-adds a point and two FP64 logarithms a draw.  So every
// score is first enclosed in FP32, [L_ik, U_ik] with the bounds derived below, and a cluster
// whose U + (largest Gumbel value) is below the best L + (smallest) is left out: it cannot
// win whatever is drawn.  If one cluster is left, it is the label.  Otherwise the ones left
// are scored in FP64, their Gumbel values are enclosed in FP32 (gumbel_approx), and FP64
// logarithms are taken for those that this cannot tell apart.  The labels are those of
// scoring and drawing everything in FP64.
// The points are taken in the order of the last counting sort, so that a warp's points
// mostly have the cluster they had in common; it is enclosed first.  Of every other cluster
// the last eight columns are tried first (W is upper triangular: column j is x_j given
// x_0 .. x_j-1, on the tightest scale where j is largest), staged in shared memory one
// cluster ahead; the few clusters that they leave standing are enclosed in full.
// Measured at d = 32, K = 20, N = 30,001: 217 us; 1518 us for every score and draw in FP64
// (with x - mu formed anew for every entry of W), 650 us with FP64 partial sums instead of
// FP32 enclosures (a warp goes on until all of its 32 points have left the cluster), 225 us
// with the clusters read from global memory where they are used (one latency after another).
//
// Enclosure: with x' = x - mu_0 and mu'_k = mu_k - mu_0 (formed in FP64, rounded to FP32,
// mu_0 the first cluster's mean: the data need not be centred), t = x' - mu' and the column
// sum y = sum_l W_l t_l in FP32, y is off by at most (d + 8) 2^-24 sum_l |W_l| (|x'_l| +
// |mu'_l|): one rounding each of W, x', mu', t, and d + 1 of the sum.  By Cauchy-Schwarz
// that is at most e = (d + 8) 2^-24 ||W_j|| (||x'|| + ||mu'||), the norms rounded up by 1%.  The
// rounding of x' and mu' in FP64, 2^-53 (|x| + |mu_0|), enters as 2^-26 (|x_l| + |mu_0l|) added
// to |x'_l|.  Sums of squares of at most 144 terms are off by 144 x 2^-24 < 1e-5 relative.
constexpr int NIW_C = 8;  // contenders a thread holds
constexpr int NIW_B = 8;  // columns at a time
constexpr int NIW_P = 8;  // clusters a thread puts off

struct Niw64 {
    int d, xs;
    int64_t N;
    const double *X, *W, *mu, *c;  // FP64 data and parameters (slots 3k)
    const float *qW, *qmu, *qn, *qc;  // FP32: W, mu - mu_0, the norms of W's columns and of mu - mu_0
    const int* idx;                // order of the points, or null
    const int* dK;
    const uint32_t* diter;
    uint64_t seed;
    int32_t* z;
};

// Dynamic shared memory, a column per thread (row stride blockDim + 1): d floats x', d floats
// t, d doubles x - mu; then the contenders: NIW_C doubles (scores) and, each of blockDim,
// NIW_C floats U, NIW_C ints, NIW_P shorts; then, per warp, two stages of NIW_B d + d floats (a cluster's
// last columns of W, mu - mu_0).
template <bool VEC>  // VEC: d is a multiple of 4, rows of the FP32 W are 16-byte aligned
__global__ void __launch_bounds__(128) labels_niw64_kernel(Niw64 a) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int K = *a.dK, d = a.d, tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, ld = nt + 1;
    double* sd = (double*)smraw + tid;                    // x - mu of the cluster in hand, FP64
    double* csc = (double*)smraw + (size_t)d * ld + tid;  // contenders' FP64 scores
    float* sx = (float*)((double*)smraw + (size_t)d * ld + NIW_C * nt);
    float* st = sx + (size_t)d * ld + tid;
    float* cu = sx + (size_t)2 * d * ld + tid;            // contenders' U, then approximate values
    int* ck = (int*)(cu - tid + NIW_C * nt) + tid;
    const int sz = (NIW_B + 1) * d, jl = (d - 1) / NIW_B * NIW_B, wl = d - jl;  // stage, last block of columns
    short* pend = (short*)(ck - tid + NIW_C * nt) + tid;
    float* stg = (float*)(pend - tid + NIW_P * nt) + (tid >> 5) * 2 * ((sz + 3) & ~3);
    auto stage = [&](int k, int b) {  // rows of NIW_B floats, then mu; one group of copies
        const float* W = a.qW + (size_t)(3 * k) * d * d + jl;
        const float* mu = a.qmu + (size_t)(3 * k) * d;
        float* to = stg + b * ((sz + 3) & ~3);
        if constexpr (VEC) {
            const int n4 = wl >> 2;  // wl is 4 or 8
            for (int e = lane; e < d * n4; e += 32) {
                const int l = n4 == 2 ? e >> 1 : e, u = n4 == 2 ? (e & 1) * 4 : 0;
                mw_cp16(to + l * NIW_B + u, W + (size_t)l * d + u);
            }
            for (int e = lane; e < d >> 2; e += 32) mw_cp16(to + d * NIW_B + 4 * e, mu + 4 * e);
        } else {
            for (int e = lane; e < d * wl; e += 32) cp_async4(to + e / wl * NIW_B + e % wl, W + (size_t)(e / wl) * d + e % wl);
            for (int e = lane; e < d; e += 32) cp_async4(to + d * NIW_B + e, mu + e);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int e = lane; e < 2 * ((sz + 3) & ~3); e += 32) stg[e] = 0.f;  // the columns beyond d
    __syncwarp();
    const Key key{a.seed, a.diter[0], a.diter[1], a.diter[2]};
    const float gam = (float)(d + 8) * 6.0e-8f * 1.02f;  // 2^-24 = 5.96e-8; the norms' 1%
    const int64_t ntiles = (a.N + nt - 1) / nt;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t p = tile * nt + tid;
        const bool live = p < a.N;  // the rest of the last block repeats the last point
        const int64_t pc = live ? p : a.N - 1, i = a.idx ? (int64_t)a.idx[pc] : pc;
        const int zi = a.z[i];
        float nx = 0.f;  // ||x'||, with the FP64 rounding's share
        __syncwarp();    // a warp stages its own 32 points, four rows at a time
        for (int r0 = 0; r0 < 32; r0 += 4) {
            int64_t ir[4];
            float n2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int u = 0; u < 4; ++u) ir[u] = __shfl_sync(0xffffffffu, i, r0 + u);
            for (int l = lane; l < d; l += 32) {
                double v[4];
                const double m0 = a.mu[l];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = a.X[ir[u] * a.xs + l];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float x = (float)(v[u] - m0), w = fabsf(x) + 1.5e-8f * (fabsf((float)v[u]) + fabsf((float)m0));
                    sx[l * ld + (tid & ~31) + r0 + u] = x;
                    n2[u] = fmaf(w, w, n2[u]);
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                for (int o = 16; o > 0; o >>= 1) n2[u] += __shfl_xor_sync(0xffffffffu, n2[u], o);
                if (lane == r0 + u) nx = sqrtf(n2[u]);
            }
        }
        __syncwarp();
        const float* x = sx + tid;
        const double* xr = a.X + i * a.xs;
        float low = -INFINITY;  // a cluster below this value cannot win
        double vb = -INFINITY;  // the best value drawn so far, and its cluster
        int kb = 0, nc = 0;
        bool drawn = false, sure = true;
        // FP64 score of cluster k
        auto score = [&](int k) -> double {
            const double* W = a.W + (size_t)(3 * k) * d * d;
            const double* mu = a.mu + (size_t)(3 * k) * d;
            double q = 0.0;
            for (int j = 0; j < d; j += 2) {  // two chains at once; each adds l = 0, 1, ... in order
                const bool two = j + 1 < d;
                sd[j * ld] = xr[j] - __ldg(mu + j);
                if (two) sd[(j + 1) * ld] = xr[j + 1] - __ldg(mu + j + 1);
                const double* Wa = W + j;
                const double* Wb = W + (two ? j + 1 : j);
                double ya = 0.0, yb = 0.0;
#pragma unroll 8
                for (int l = 0; l <= j; ++l) {
                    const double t = sd[l * ld];
                    ya = fma(__ldg(Wa + l * d), t, ya);
                    yb = fma(__ldg(Wb + l * d), t, yb);
                }
                q = fma(ya, ya, q);
                if (two) {
                    yb = fma(__ldg(Wb + (j + 1) * d), sd[(j + 1) * ld], yb);
                    q = fma(yb, yb, q);
                }
            }
            return __ldg(a.c + 3 * k) - 0.5 * q;
        };
        // the contenders' FP64 values against the best one drawn (ties to the lower index)
        auto draw_all = [&]() {
            for (int e = 0; e < nc; ++e) {
                const int k = ck[e * nt];
                uint32_t w[4];
                key.block((uint32_t)i, TAG_Z, (uint32_t)(k >> 1), w);
                const double v = csc[e * nt] + ((k & 1) ? gumbel_of<double>(w[2], w[3]) : gumbel_of<double>(w[0], w[1]));
                if (v > vb || (v == vb && drawn && k < kb)) {
                    vb = v;
                    kb = k;
                    drawn = true;
                }
            }
            nc = 0;
        };
        auto purge = [&]() {  // contenders that later bounds have ruled out
            int m = 0;
            for (int e = 0; e < nc; ++e) {
                if (cu[e * nt] + 37.5f < low) continue;
                cu[m * nt] = cu[e * nt];
                ck[m * nt] = ck[e * nt];
                ++m;
            }
            nc = m;
        };
        auto score_all = [&]() {  // FP64 scores of the contenders; those without a value are dropped
            int m = 0;
            for (int e = 0; e < nc; ++e) {
                const int k = ck[e * nt];
                const double sc = score(k);
                if (!(sc > -INFINITY)) continue;
                csc[m * nt] = sc;
                ck[m * nt] = k;
                ++m;
            }
            nc = m;
        };
        auto bound = [&](float c) {  // a sum of squares above it leaves cluster k (weight and determinant c) out
            return 2.f * (c + 37.5f - low + 1e-3f + 1e-6f * fabsf(c)) * 1.00002f + 1e-2f;
        };
        auto square = [&](float y, float e, float& qlo, float& qhi) {
            const float h = fabsf(y) + e, g = fmaxf(fabsf(y) - e, 0.f);
            qlo = fmaf(g, g, qlo);
            qhi = fmaf(h, h, qhi);
        };
        auto admit = [&](int k, float c, float qlo, float qhi) {
            const float slack = 1e-3f + 1e-6f * fabsf(c);
            float U = c - 0.5f * (qlo * 0.99998f) + slack;
            float L = c - 0.5f * (qhi * 1.00002f) - slack;
            if (!(fabsf(U) < INFINITY)) {  // c or a square left FP32's range
                if (!(__ldg(a.c + 3 * k) > -INFINITY)) return;  // weight zero, or NaN
                U = INFINITY;
            }
            if (U + 37.5f < low) return;
            if (!(fabsf(L) < INFINITY)) {  // nothing known: FP64 decides
                L = -INFINITY;
                sure = false;
            }
            if (nc == NIW_C) {
                purge();
                if (nc == NIW_C) {
                    score_all();
                    draw_all();
                    if (drawn) low = fmaxf(low, (float)vb - 1e-3f - 1e-6f * fabsf((float)vb));
                }
            }
            cu[nc * nt] = U;
            ck[nc * nt] = k;
            ++nc;
            low = fmaxf(low, L - 3.7f);
        };
        auto enclose = [&](int k) {  // every column
            const float* W = a.qW + (size_t)(3 * k) * d * d;
            const float* mu = a.qmu + (size_t)(3 * k) * d;
            const float* qn = a.qn + (size_t)(3 * k) * d;
            const float c = (float)__ldg(a.c + 3 * k), thr = bound(c);
#pragma unroll 8
            for (int l = 0; l < d; ++l) st[l * ld] = x[l * ld] - __ldg(mu + l);
            const float ga = gam * (nx + __ldg(a.qc + 3 * k));
            float qlo = 0.f, qhi = 0.f;
            for (int j0 = jl; j0 >= 0; j0 -= NIW_B) {
                float y[NIW_B];
#pragma unroll
                for (int u = 0; u < NIW_B; ++u) y[u] = 0.f;
                const int le = min(d, j0 + NIW_B);
#pragma unroll 8
                for (int l = 0; l < le; ++l) {
                    const float t = st[l * ld];
                    float w[NIW_B];
                    if constexpr (VEC) {
#pragma unroll
                        for (int u = 0; u < NIW_B; u += 4) {
                            const float4 v = j0 + u < d ? __ldg((const float4*)(W + l * d + j0 + u)) : make_float4(0.f, 0.f, 0.f, 0.f);
                            w[u] = v.x;
                            w[u + 1] = v.y;
                            w[u + 2] = v.z;
                            w[u + 3] = v.w;
                        }
                    } else {
#pragma unroll
                        for (int u = 0; u < NIW_B; ++u) w[u] = j0 + u < d ? __ldg(W + l * d + j0 + u) : 0.f;
                    }
#pragma unroll
                    for (int u = 0; u < NIW_B; ++u) y[u] = fmaf(l <= j0 + u ? w[u] : 0.f, t, y[u]);
                }
#pragma unroll
                for (int u = 0; u < NIW_B; ++u)
                    if (j0 + u < d) square(y[u], ga * __ldg(qn + j0 + u), qlo, qhi);
                if (qlo > thr && qlo < INFINITY) return;  // a sum that overflowed bounds nothing
            }
            admit(k, c, qlo, qhi);
        };
        const int hint = zi >= 0 && zi < K ? zi : 0;
        int np = 1;
        pend[0] = (short)hint;
        stage(0, 0);
        // clusters put off are enclosed in full with the lanes' own ones side by side: the
        // point's own first of all, the others when a thread holds no more, and at the end
        for (int k = -1; k <= K; ++k) {
            if (k < 0 || k == K || np == NIW_P)
                while (np > 0) enclose(pend[--np * nt]);
            if (k < 0 || k == K) continue;
            const float c = (float)__ldg(a.c + 3 * k), mn = __ldg(a.qc + 3 * k);
            float en[NIW_B];
#pragma unroll
            for (int u = 0; u < NIW_B; ++u) en[u] = u < wl ? __ldg(a.qn + (size_t)(3 * k) * d + jl + u) : 0.f;
            if (k + 1 < K) {
                stage(k + 1, (k + 1) & 1);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncwarp();
            const float* Wl = stg + (k & 1) * ((sz + 3) & ~3);
            const float* ml = Wl + d * NIW_B;
            float y[NIW_B];
#pragma unroll
            for (int u = 0; u < NIW_B; ++u) y[u] = 0.f;
#pragma unroll 8
            for (int l = 0; l < jl; ++l) {
                const float t = x[l * ld] - ml[l];
                const float4 w0 = *(const float4*)(Wl + l * NIW_B), w1 = *(const float4*)(Wl + l * NIW_B + 4);
                y[0] = fmaf(w0.x, t, y[0]);
                y[1] = fmaf(w0.y, t, y[1]);
                y[2] = fmaf(w0.z, t, y[2]);
                y[3] = fmaf(w0.w, t, y[3]);
                y[4] = fmaf(w1.x, t, y[4]);
                y[5] = fmaf(w1.y, t, y[5]);
                y[6] = fmaf(w1.z, t, y[6]);
                y[7] = fmaf(w1.w, t, y[7]);
            }
#pragma unroll
            for (int v = 0; v < NIW_B; ++v)
                if (v < wl) {
                    const float t = x[(jl + v) * ld] - ml[jl + v];
#pragma unroll
                    for (int u = v; u < NIW_B; ++u) y[u] = fmaf(Wl[(jl + v) * NIW_B + u], t, y[u]);
                }
            const float ga = gam * (nx + mn);
            float qlo = 0.f, qhi = 0.f;
#pragma unroll
            for (int u = 0; u < NIW_B; ++u)
                if (u < wl) square(y[u], ga * en[u], qlo, qhi);
            if (k != hint && !(qlo > bound(c) && qlo < INFINITY)) pend[np++ * nt] = (short)k;
            __syncwarp();  // the stage is filled again
        }
        purge();
        if (nc == 1 && !drawn && sure) {
            kb = ck[0];
        } else if (nc > 0) {
            score_all();
            double vmax = vb;
            for (int e = 0; e < nc; ++e) {
                const int k = ck[e * nt];
                uint32_t w[4];
                key.block((uint32_t)i, TAG_Z, (uint32_t)(k >> 1), w);
                const float g = (k & 1) ? gumbel_approx(w[2], w[3]) : gumbel_approx(w[0], w[1]);
                cu[e * nt] = g;
                vmax = fmax(vmax, csc[e * nt] + (double)g);
            }
            const double cut = vmax - approx_margin(fabs(vmax));
            int m = 0;  // the contenders that the approximation cannot tell from the best
            for (int e = 0; e < nc; ++e)
                if (csc[e * nt] + (double)cu[e * nt] >= cut) {
                    csc[m * nt] = csc[e * nt];
                    ck[m * nt] = ck[e * nt];
                    ++m;
                }
            nc = m;
            if (nc == 1 && !(drawn && vb >= cut)) kb = ck[0];
            else draw_all();
        }
        if (live) a.z[i] = kb;
    }
}

// ------------------------------------------------------------------ counting sort
// Stable counting sort of the points by cluster (the order the statistics step visits
// them in), in tiles of SORT_TILE points: four rounds of 256, one point per thread per
// round, so that a tile's points are ranked in index order (round, warp, lane).
__global__ void hist_kernel(const int32_t* z, int64_t N, int T_tiles, int Kmax, const int* gate, int* hist) {
    if (gate && *gate == 0) return;
    extern __shared__ int cnt[];
    const int t = blockIdx.x;
    for (int k = threadIdx.x; k < Kmax; k += blockDim.x) cnt[k] = 0;
    int zq[SORT_TILE / 256];
#pragma unroll
    for (int q = 0; q < SORT_TILE / 256; ++q) {
        const int64_t i = (int64_t)t * SORT_TILE + q * 256 + threadIdx.x;
        zq[q] = i < N ? z[i] : -1;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < SORT_TILE / 256; ++q)
        if ((unsigned)zq[q] < (unsigned)Kmax) atomicAdd(&cnt[zq[q]], 1);  // labels are always in range
    __syncthreads();
    for (int k = threadIdx.x; k < Kmax; k += blockDim.x) hist[(size_t)k * T_tiles + t] = cnt[k];
}

// Exclusive scan of each cluster's row of tile counts (block k), row total into tot[k];
// the last block to finish turns the totals into the clusters' starts (exclusive prefix,
// tot[K] = N) and re-arms the counter *done for the next launch.
__global__ void scan_kernel(int* hist, int T_tiles, const int* dK, const int* gate, int* tot, int* done) {
    if (gate && *gate == 0) return;
    const int k = blockIdx.x, K = *dK;
    __shared__ int wsum[32];
    __shared__ int s_last;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (k < K) {
        int* row = hist + (size_t)k * T_tiles;
        const int per = (T_tiles + blockDim.x - 1) / blockDim.x;
        const int a = threadIdx.x * per, b = min(T_tiles, a + per);
        int s = 0;
        for (int t = a; t < b; ++t) s += row[t];
        // block exclusive scan of s
        int x = s;
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[w] = x;
        __syncthreads();
        if (w == 0) {
            int nw = blockDim.x >> 5;
            int v = lane < nw ? wsum[lane] : 0;
            for (int o = 1; o < 32; o <<= 1) {
                int y = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += y;
            }
            if (lane < nw) wsum[lane] = v;
        }
        __syncthreads();
        int excl = x - s + (w > 0 ? wsum[w - 1] : 0);
        for (int t = a; t < b; ++t) {
            int v = row[t];
            row[t] = excl;
            excl += v;
        }
        if (threadIdx.x == blockDim.x - 1) {
            tot[k] = excl;
            __threadfence();
        }
    } else if (threadIdx.x == 0) {
        tot[k] = 0;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(done, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last || w != 0) return;
    __threadfence();
    int acc = 0;
    for (int k0 = 0; k0 < K; k0 += 32) {
        const int v = k0 + lane < K ? __ldcg(tot + k0 + lane) : 0;
        int x = v;
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (k0 + lane < K) tot[k0 + lane] = acc + x - v;
        acc += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) {
        tot[K] = acc;
        *done = 0;
    }
}

__global__ void scatter_kernel(const int32_t* z, int64_t N, int T_tiles, const int* hist, const int* starts,
                               const int* gate, int Kmax, int* idx) {
    if (gate && *gate == 0) return;
    extern __shared__ int wc[];  // 8 warps x Kmax counts of the round, then Kmax running bases
    int* base = wc + 8 * Kmax;
    const int t = blockIdx.x;
    for (int e = threadIdx.x; e < 8 * Kmax; e += blockDim.x) wc[e] = 0;
    for (int k = threadIdx.x; k < Kmax; k += blockDim.x) base[k] = starts[k] + hist[(size_t)k * T_tiles + t];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int zq[SORT_TILE / 256];
#pragma unroll
    for (int q = 0; q < SORT_TILE / 256; ++q) {
        const int64_t i = (int64_t)t * SORT_TILE + q * 256 + threadIdx.x;
        zq[q] = i < N ? z[i] : -1;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < SORT_TILE / 256; ++q) {
        const int64_t i = (int64_t)t * SORT_TILE + q * 256 + threadIdx.x;
        const bool live = (unsigned)zq[q] < (unsigned)Kmax;  // labels are always in range
        const int k = live ? zq[q] : -1 - lane;             // dead lanes never match live ones
        const unsigned m = __match_any_sync(0xffffffffu, k);
        const int r = __popc(m & ((1u << lane) - 1u));
        if (live && r == 0) wc[w * Kmax + k] = __popc(m);
        __syncthreads();
        if (live) {
            int before = 0;
            for (int v = 0; v < w; ++v) before += wc[v * Kmax + k];
            idx[base[k] + before + r] = (int)i;
        }
        __syncthreads();
        // the bases move past this round's points; the counts are cleared for the next
        for (int kk = threadIdx.x; kk < Kmax; kk += blockDim.x) {
            int s = 0;
            for (int v = 0; v < 8; ++v) {
                s += wc[v * Kmax + kk];
                wc[v * Kmax + kk] = 0;
            }
            base[kk] += s;
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ sub-labels + stats
// Starts of the runs of equal labels among kq[0..np) (np <= blockDim), by warp ballots:
// runs[0..n) are the starts, runs[n] = np, *nruns = n.  All threads must call it.
__device__ inline void find_runs(const int* kq, int np, int* runs, int* nruns, int* wcnt) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = (blockDim.x + 31) >> 5;
    const bool f = tid < np && (tid == 0 || kq[tid] != kq[tid - 1]);
    const unsigned m = __ballot_sync(0xffffffffu, f);
    if (lane == 0) wcnt[w] = __popc(m);
    __syncthreads();
    int before = 0, total = 0;
    for (int v = 0; v < nw; ++v) {
        if (v < w) before += wcnt[v];
        total += wcnt[v];
    }
    if (f) runs[before + __popc(m & ((1u << lane) - 1u))] = tid;
    if (tid == 0) {
        runs[total] = np;
        *nruns = total;
    }
    __syncthreads();
}


template <typename T>
struct SubArgs {
    int kind, d, xs;
    int64_t N;
    const void* X;
    ParamView<T> pv;
    const T* shift;  // K_max x d, storage coordinates
    const int32_t* z;
    uint8_t* zbar;
    const int* idx;
    const int* dK;
    const uint32_t* diter;
    const int* gate;
    uint64_t seed;
    int draw;        // 1: draw z-bar; 0: keep
    int P;           // points per tile
    int G;           // point groups per block
    int64_t R;       // points per CTA
    StatLayout L;
    double* rec;     // (G2 + K_max) x 2 x E
};

template <typename T, typename XT>
__device__ inline T sub_score(const SubArgs<T>& a, int s, const T* xr) {
    const int d = a.d;
    if (a.kind == DPMM_PRIOR_NIW) {
        const T* W = a.pv.W + (size_t)s * d * d;
        const T* mu = a.pv.mu + (size_t)s * d;
        T q = 0;
        for (int j = 0; j < d; ++j) {
            T y = 0;
            for (int l = 0; l <= j; ++l) y += __ldg(W + l * d + j) * (xr[l] - __ldg(mu + l));
            q += y * y;
        }
        return __ldg(a.pv.c + s) - (T)0.5 * q;
    }
    const T* lt = a.pv.lt + (size_t)s * d;
    T acc = 0;
    for (int j = 0; j < d; ++j) acc += xr[j] * __ldg(lt + j);
    return __ldg(a.pv.c + s) + acc;
}

// Dynamic shared memory: P x dp T (point rows), P ints (k), P bytes (h), then the
// flush buffer G x nblk x 32 T.
template <typename T, typename XT, int MAXT>
__global__ void __launch_bounds__(MAXT) substats_kernel(SubArgs<T> a) {
    if (a.gate && *a.gate == 0) return;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int d = a.d, dp = a.L.dp, P = a.P, G = a.G, nblk = a.L.nblk;
    T* xs = (T*)smraw;
    int* kq = (int*)(xs + (size_t)P * dp);
    int* runs = kq + P;          // run starts, P + 1
    int* nruns = runs + P + 1;
    unsigned char* hq = (unsigned char*)(nruns + 1);
    T* red = (T*)(smraw + (((size_t)P * dp * sizeof(T) + (2 * P + 2) * sizeof(int) + P + 15) / 16) * 16);

    const int tid = threadIdx.x, nt = blockDim.x;
    const int g = blockIdx.x;
    const int64_t p0 = (int64_t)g * a.R, p1 = min(a.N, p0 + a.R);
    Key key{a.seed, a.diter[0], a.diter[1], a.diter[2]};
    const XT* X = (const XT*)a.X;

    // register block of this thread
    const bool worker = tid < nblk * G;
    const int myblk = worker ? tid % nblk : 0, grp = worker ? tid / nblk : 0;
    int jb = 0, lb = 0;
    a.L.blk_coords(myblk, jb, lb);
    T acc[16], accr[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) acc[e] = accr[e] = 0;
    int cur = -1;

    auto flush = [&](int k) {
        __syncthreads();
        if (worker) {
            T* r = red + ((size_t)grp * nblk + myblk) * 32;
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                r[e] = acc[e];
                r[16 + e] = accr[e];
            }
        }
        __syncthreads();
        double* out = a.rec + (size_t)(g + k) * 2 * a.L.E;
        for (int e = tid; e < nblk * 16; e += nt) {
            int b = e >> 4, q = e & 15;
            double all = 0.0, rr = 0.0;
            for (int gg = 0; gg < G; ++gg) {
                all += (double)red[((size_t)gg * nblk + b) * 32 + q];
                rr += (double)red[((size_t)gg * nblk + b) * 32 + 16 + q];
            }
            out[b * 16 + q] = all;            // sub-cluster l
            out[a.L.E + b * 16 + q] = rr;     // sub-cluster r
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) acc[e] = accr[e] = 0;
    };

    for (int64_t base = p0; base < p1; base += P) {
        const int np = (int)min((int64_t)P, p1 - base);
        __syncthreads();
        if (tid < np) {
            const int i = a.idx[base + tid];
            const int k = a.z[i];
            T* xr = xs + (size_t)tid * dp;
            for (int j = 0; j < d; ++j) xr[j] = ldx<T, XT>(X + (int64_t)i * a.xs + j);
            int h;
            if (a.draw) {
                uint32_t w[4];
                key.block((uint32_t)i, TAG_ZBAR, 0, w);
                const T sl = sub_score<T, XT>(a, 3 * k + 1, xr), sr = sub_score<T, XT>(a, 3 * k + 2, xr);
                bool near = true;  // FP64: an FP32 Gumbel difference decides where it can
                if constexpr (sizeof(T) == 8) {
                    const T diff = (sr - sl) + (T)(gumbel_approx(w[2], w[3]) - gumbel_approx(w[0], w[1]));
                    near = !(fabs(diff) > approx_margin(fabs(sl) + fabs(sr)));
                    h = diff > 0 ? 1 : 0;
                }
                if (near) h = sr + gumbel_of<T>(w[2], w[3]) > sl + gumbel_of<T>(w[0], w[1]) ? 1 : 0;
                a.zbar[i] = (uint8_t)h;
            } else {
                h = a.zbar[i];
            }
            const T* sh = a.shift + (size_t)k * d;
            for (int j = 0; j < d; ++j) xr[j] -= sh[j];
            xr[d] = 1;
            for (int j = d + 1; j < dp; ++j) xr[j] = 0;
            kq[tid] = k;
            hq[tid] = (unsigned char)h;
        }
        __syncthreads();
        {
            __shared__ int wcnt[32];
            find_runs(kq, np, runs, nruns, wcnt);
        }
        const int nr = *nruns;
        for (int r = 0; r < nr; ++r) {
            const int qs = runs[r], qe = runs[r + 1];
            const int k = kq[qs];
            if (k != cur) {
                if (cur >= 0) flush(cur);
                cur = k;
            }
            if (worker) {
                for (int q = qs + grp; q < qe; q += G) {
                    const T* xr = xs + (size_t)q * dp;
                    T xj[4], xl[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        xj[u] = xr[jb * 4 + u];
                        xl[u] = xr[lb * 4 + u];
                    }
                    if (hq[q]) {
#pragma unroll
                        for (int u = 0; u < 4; ++u)
#pragma unroll
                            for (int v = 0; v < 4; ++v) accr[u * 4 + v] = fma(xj[u], xl[v], accr[u * 4 + v]);
                    } else {
#pragma unroll
                        for (int u = 0; u < 4; ++u)
#pragma unroll
                            for (int v = 0; v < 4; ++v) acc[u * 4 + v] = fma(xj[u], xl[v], acc[u * 4 + v]);
                    }
                }
            }
        }
    }
    if (cur >= 0) flush(cur);
}

// Gaussian FP64 sub-labels and statistics.  What bounds the step is the FP64 pipe (two lanes
// an SM): the two sub-cluster scores take d^2 FP64 multiply-adds a point, the sums d^2 / 2.
// So the scores are enclosed in FP32 first, as in labels_niw64_kernel (the bounds are derived
// there), and so are the two Gumbel values; only the points whose sub-label these enclosures
// leave open are scored in FP64, a warp to each (lane j takes column j, adding l = 0, 1, ... in
// order), so that the sub-labels are those of scoring every point in FP64.  The sums are FP64.
// Measured at d = 32, K = 20, N = 30,001: 107 us per step; 250 us with every score in FP64,
// 759 us so and in 59 ranges of 512 points, on 59 of 152 SMs.
// Dynamic shared memory: P x dp doubles (rows), P floats (norms), P x 4 floats (enclosures),
// P ints (k), P + 2 ints (runs), P + 1 ints (points left open), P bytes (h), then d x (P + 1)
// floats (x - mu_0 by coordinate), later the flush buffer G x nblk x 32 doubles.
struct Sub64 {
    SubArgs<double> a;
    const float *qW, *qmu, *qn, *qc;  // FP32: W, mu - mu_0, the norms of W's columns and of mu - mu_0
};

__host__ __device__ inline size_t sub64_head(int P, int dp) {
    return ((size_t)P * dp * 8 + (size_t)P * 20 + (size_t)(3 * P + 3) * 4 + P + 15) / 16 * 16;
}

template <int MAXT>
__global__ void __launch_bounds__(MAXT) substats_niw64_kernel(Sub64 b) {
    const SubArgs<double>& a = b.a;
    if (a.gate && *a.gate == 0) return;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int d = a.d, dp = a.L.dp, P = a.P, G = a.G, nblk = a.L.nblk;
    double* xs = (double*)smraw;
    float* nrm = (float*)(xs + (size_t)P * dp);
    float* enc = nrm + P;        // lower and upper bound of each sub-cluster's score
    int* kq = (int*)(enc + 4 * P);
    int* runs = kq + P;          // run starts, P + 1
    int* nruns = runs + P + 1;
    int* open = nruns + 1;       // points whose sub-label FP64 decides; the count at P
    unsigned char* hq = (unsigned char*)(open + P + 1);
    double* red = (double*)(smraw + sub64_head(P, dp));
    float* xf = (float*)red;     // used before any flush of the same batch
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
    const int g = blockIdx.x, ldf = P + 1;
    const int64_t p0 = (int64_t)g * a.R, p1 = min(a.N, p0 + a.R);
    const Key key{a.seed, a.diter[0], a.diter[1], a.diter[2]};
    const double* X = (const double*)a.X;
    const float gam = (float)(d + 8) * 6.0e-8f * 1.02f;
    __shared__ int wcnt[32];

    const bool worker = tid < nblk * G;
    const int myblk = worker ? tid % nblk : 0, grp = worker ? tid / nblk : 0;
    int jb = 0, lb = 0;
    a.L.blk_coords(myblk, jb, lb);
    double acc[16], accr[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) acc[e] = accr[e] = 0.0;
    int cur = -1;

    auto flush = [&](int k) {
        __syncthreads();
        if (worker) {
            double* r = red + ((size_t)grp * nblk + myblk) * 32;
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                r[e] = acc[e];
                r[16 + e] = accr[e];
            }
        }
        __syncthreads();
        double* out = a.rec + (size_t)(g + k) * 2 * a.L.E;
        for (int e = tid; e < nblk * 16; e += nt) {
            const int bl = e >> 4, q = e & 15;
            double sl = 0.0, sr = 0.0;
            for (int gg = 0; gg < G; ++gg) {
                sl += red[((size_t)gg * nblk + bl) * 32 + q];
                sr += red[((size_t)gg * nblk + bl) * 32 + 16 + q];
            }
            out[bl * 16 + q] = sl;
            out[a.L.E + bl * 16 + q] = sr;
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) acc[e] = accr[e] = 0.0;
    };

    for (int64_t base = p0; base < p1; base += P) {
        const int np = (int)min((int64_t)P, p1 - base);
        __syncthreads();
        for (int r = warp; r < np; r += nt >> 5) {  // one warp per row
            const int i = a.idx[base + r];
            float n2 = 0.f;
            for (int l = lane; l < d; l += 32) {
                const double v = X[(int64_t)i * a.xs + l];
                xs[(size_t)r * dp + l] = v;
                if (a.draw) {
                    const double m0 = a.pv.mu[l];
                    const float x = (float)(v - m0), w = fabsf(x) + 1.5e-8f * (fabsf((float)v) + fabsf((float)m0));
                    xf[l * ldf + r] = x;
                    n2 = fmaf(w, w, n2);
                }
            }
            if (a.draw) {
                for (int o = 16; o > 0; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
                if (lane == 0) nrm[r] = sqrtf(n2);
            }
            if (lane == 0) kq[r] = a.z[i];
        }
        if (tid == 0) open[P] = 0;
        __syncthreads();
        if (a.draw) {
            for (int it = tid; it < 2 * np; it += nt) {  // enclosure of sub-cluster h's score of point p
                const int h = it >= np, p = it - (h ? np : 0), s = 3 * kq[p] + 1 + h;
                const float* W = b.qW + (size_t)s * d * d;
                const float* mu = b.qmu + (size_t)s * d;
                const float* qn = b.qn + (size_t)s * d;
                const float ga = gam * (nrm[p] + __ldg(b.qc + s));
                const float* x = xf + p;
                float qlo = 0.f, qhi = 0.f;
                for (int j0 = 0; j0 < d; j0 += 4) {
                    float y[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
                    for (int l = 0; l < min(d, j0 + 4); ++l) {
                        const float t = x[l * ldf] - __ldg(mu + l);
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            y[u] = fmaf(l <= j0 + u && j0 + u < d ? __ldg(W + l * d + j0 + u) : 0.f, t, y[u]);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (j0 + u < d) {
                            const float e = ga * __ldg(qn + j0 + u), hi = fabsf(y[u]) + e, lo = fmaxf(fabsf(y[u]) - e, 0.f);
                            qlo = fmaf(lo, lo, qlo);
                            qhi = fmaf(hi, hi, qhi);
                        }
                }
                const float c = (float)__ldg(a.pv.c + s), slack = 1e-3f + 1e-6f * fabsf(c);
                enc[4 * p + 2 * h] = c - 0.5f * (qhi * 1.00002f) - slack;
                enc[4 * p + 2 * h + 1] = c - 0.5f * (qlo * 0.99998f) + slack;
            }
            __syncthreads();
        }
        for (int p = tid; p < np; p += nt) {
            const int i = a.idx[base + p];
            int h = 0;
            if (a.draw) {
                uint32_t w[4];
                key.block((uint32_t)i, TAG_ZBAR, 0, w);
                const float dg = gumbel_approx(w[2], w[3]) - gumbel_approx(w[0], w[1]);
                const float lo = enc[4 * p + 2] - enc[4 * p + 1] + dg, hi = enc[4 * p + 3] - enc[4 * p] + dg;
                const float m = 1e-3f + 1e-6f * (fabsf(enc[4 * p]) + fabsf(enc[4 * p + 2]));  // the sums' own rounding
                if (lo > m) h = 1;
                else if (hi < -m) h = 0;
                else open[atomicAdd(&open[P], 1)] = p;
                a.zbar[i] = (uint8_t)h;
            } else {
                h = a.zbar[i];
            }
            hq[p] = (unsigned char)h;
        }
        __syncthreads();
        if (a.draw) {
            const int no = open[P];
            for (int o = warp; o < no; o += nt >> 5) {
                const int p = open[o], k = kq[p], i = a.idx[base + p];
                const double* x = xs + (size_t)p * dp;
                const double* W0 = a.pv.W + (size_t)(3 * k + 1) * d * d;
                const double* m0 = a.pv.mu + (size_t)(3 * k + 1) * d;
                double q0 = 0.0, q1 = 0.0;
                for (int j0 = 0; j0 < d; j0 += 32) {
                    const int j = min(j0 + lane, d - 1);
                    double y0 = 0.0, y1 = 0.0;
                    for (int l = 0; l < min(d, j0 + 32); ++l) {
                        const double t0 = x[l] - __ldg(m0 + l), t1 = x[l] - __ldg(m0 + d + l);
                        if (l <= j) {
                            y0 = fma(__ldg(W0 + l * d + j), t0, y0);
                            y1 = fma(__ldg(W0 + (size_t)d * d + l * d + j), t1, y1);
                        }
                    }
                    for (int u = 0; u < min(32, d - j0); ++u) {
                        const double v0 = __shfl_sync(0xffffffffu, y0, u), v1 = __shfl_sync(0xffffffffu, y1, u);
                        q0 = fma(v0, v0, q0);
                        q1 = fma(v1, v1, q1);
                    }
                }
                if (lane == 0) {
                    uint32_t w[4];
                    key.block((uint32_t)i, TAG_ZBAR, 0, w);
                    const double sl = a.pv.c[3 * k + 1] - 0.5 * q0, sr = a.pv.c[3 * k + 2] - 0.5 * q1;
                    const double diff = (sr - sl) + (double)(gumbel_approx(w[2], w[3]) - gumbel_approx(w[0], w[1]));
                    int h = diff > 0 ? 1 : 0;
                    if (!(fabs(diff) > approx_margin(fabs(sl) + fabs(sr))))
                        h = sr + gumbel_of<double>(w[2], w[3]) > sl + gumbel_of<double>(w[0], w[1]) ? 1 : 0;
                    a.zbar[i] = (uint8_t)h;
                    hq[p] = (unsigned char)h;
                }
            }
            __syncthreads();  // the rows are still read above
        }
        for (int e = tid; e < np * dp; e += nt) {  // the row less the cluster's centre, then 1, then zeros
            const int p = e / dp, j = e % dp;
            xs[e] = j < d ? xs[e] - a.shift[(size_t)kq[p] * d + j] : (j == d ? 1.0 : 0.0);
        }
        __syncthreads();
        find_runs(kq, np, runs, nruns, wcnt);
        const int nr = *nruns;
        for (int r = 0; r < nr; ++r) {
            const int qs = runs[r], qe = runs[r + 1];
            const int k = kq[qs];
            if (k != cur) {
                if (cur >= 0) flush(cur);
                cur = k;
            }
            if (worker) {
                for (int q = qs + grp; q < qe; q += G) {
                    const double* xr = xs + (size_t)q * dp;
                    double xj[4], xl[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        xj[u] = xr[jb * 4 + u];
                        xl[u] = xr[lb * 4 + u];
                    }
                    if (hq[q]) {
#pragma unroll
                        for (int u = 0; u < 4; ++u)
#pragma unroll
                            for (int v = 0; v < 4; ++v) accr[u * 4 + v] = fma(xj[u], xl[v], accr[u * 4 + v]);
                    } else {
#pragma unroll
                        for (int u = 0; u < 4; ++u)
#pragma unroll
                            for (int v = 0; v < 4; ++v) acc[u * 4 + v] = fma(xj[u], xl[v], acc[u * 4 + v]);
                    }
                }
            }
        }
    }
    if (cur >= 0) flush(cur);
}

// FP32 variant for d <= DV (DV = 32 or 64): the sub-cluster parameters of the current
// cluster run are staged in shared memory (factor transposed and zero-padded to
// DV x DV, so row j holds W[l][j] for l <= j), the point's x - mu sits in registers,
// and each sub-cluster score costs d(d+1)/2 FMAs fed by float4 broadcast loads.
// Statistics: one 4x4 register block per worker thread and one accumulator set per
// sub-cluster (the branch on h is uniform within a warp: a warp's lanes share the
// point).  Dynamic shared memory: P x dp point rows, P ints (k), P + 2 ints (runs),
// P bytes (h), then 2 DV x DV + 2 DV + 2 + d floats (staged parameters), then the
// flush buffer G x nblk x 32 floats.
template <int DV, typename XT>
__global__ void __launch_bounds__(256) substats_f32_kernel(SubArgs<float> a) {
    if (a.gate && *a.gate == 0) return;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int d = a.d, dp = a.L.dp, P = a.P, G = a.G, nblk = a.L.nblk;
    float* xs = (float*)smraw;
    int* kq = (int*)(xs + (size_t)P * dp);
    int* runs = kq + P;
    int* nruns = runs + P + 1;
    unsigned char* hq = (unsigned char*)(nruns + 1);
    float* stg = (float*)(smraw + (((size_t)P * dp * 4 + (2 * P + 2) * sizeof(int) + P + 15) / 16) * 16);
    float* WT0 = stg;                 // DV x DV
    float* WT1 = WT0 + DV * DV;       // DV x DV
    float* mu0 = WT1 + DV * DV;       // DV
    float* mu1 = mu0 + DV;            // DV
    float* cc = mu1 + DV;             // 2
    float* shf = cc + 2;              // d (cluster shift)
    float* red = (float*)(((uintptr_t)(shf + DV) + 15) & ~(uintptr_t)15);
    __shared__ int staged;

    const int tid = threadIdx.x, nt = blockDim.x;
    const int g = blockIdx.x;
    const int64_t p0 = (int64_t)g * a.R, p1 = min(a.N, p0 + a.R);
    Key key{a.seed, a.diter[0], a.diter[1], a.diter[2]};
    const XT* X = (const XT*)a.X;
    const bool worker = tid < nblk * G;
    const int myblk = worker ? tid % nblk : 0, grp = worker ? tid / nblk : 0;
    int jb = 0, lb = 0;
    a.L.blk_coords(myblk, jb, lb);
    float acc0[16], acc1[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) acc0[e] = acc1[e] = 0.f;
    int cur = -1;
    if (tid == 0) staged = -1;

    auto flush = [&](int k) {
        __syncthreads();
        if (worker) {
            float* r = red + ((size_t)grp * nblk + myblk) * 32;
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                r[e] = acc0[e];
                r[16 + e] = acc1[e];
            }
        }
        __syncthreads();
        double* out = a.rec + (size_t)(g + k) * 2 * a.L.E;
        for (int e = tid; e < nblk * 16; e += nt) {
            int b = e >> 4, q = e & 15;
            double s0 = 0.0, s1 = 0.0;
            for (int gg = 0; gg < G; ++gg) {
                s0 += (double)red[((size_t)gg * nblk + b) * 32 + q];
                s1 += (double)red[((size_t)gg * nblk + b) * 32 + 16 + q];
            }
            out[b * 16 + q] = s0;
            out[a.L.E + b * 16 + q] = s1;
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) acc0[e] = acc1[e] = 0.f;
    };

    for (int64_t base = p0; base < p1; base += P) {
        const int np = (int)min((int64_t)P, p1 - base);
        __syncthreads();
        int i = 0;
        float v[DV];
        if (tid < np) {
            i = a.idx[base + tid];
            kq[tid] = a.z[i];
            if constexpr (sizeof(XT) == 4) {  // rows are 16-byte aligned (stride a multiple of 4 floats)
                const float4* xr4 = (const float4*)(X + (int64_t)i * a.xs);
#pragma unroll
                for (int j4 = 0; j4 < DV / 4; ++j4) {
                    const float4 q = j4 * 4 < d ? xr4[j4] : make_float4(0.f, 0.f, 0.f, 0.f);
                    v[4 * j4] = q.x;
                    v[4 * j4 + 1] = q.y;
                    v[4 * j4 + 2] = q.z;
                    v[4 * j4 + 3] = q.w;
                }
#pragma unroll
                for (int j = 0; j < DV; ++j)
                    if (j >= d) v[j] = 0.f;
            } else {
#pragma unroll
                for (int j = 0; j < DV; ++j) v[j] = j < d ? ldx<float, XT>(X + (int64_t)i * a.xs + j) : 0.f;
            }
        }
        __syncthreads();
        {
            __shared__ int wcnt2[32];
            find_runs(kq, np, runs, nruns, wcnt2);
        }
        const int nr = *nruns;
        for (int r = 0; r < nr; ++r) {
            const int qs = runs[r], qe = runs[r + 1];
            const int k = kq[qs];
            if (k != staged) {  // uniform: stage this cluster's two sub-clusters
                __syncthreads();
                for (int e = tid; e < 2 * DV * DV; e += nt) {
                    const int h = e / (DV * DV), jj = (e / DV) % DV, l = e % DV;
                    const int s = 3 * k + 1 + h;
                    stg[e] = (jj < d && l <= jj) ? a.pv.W[((size_t)s * d + l) * d + jj] : 0.f;
                }
                for (int e = tid; e < 2 * DV; e += nt) {
                    const int h = e / DV, j = e % DV;
                    mu0[e] = j < d ? a.pv.mu[(size_t)(3 * k + 1 + h) * d + j] : 0.f;
                }
                if (tid < 2) cc[tid] = a.pv.c[3 * k + 1 + tid];
                for (int j = tid; j < d; j += nt) shf[j] = a.shift[(size_t)k * d + j];
                __syncthreads();
                if (tid == 0) staged = k;
            }
            if (tid >= qs && tid < qe) {
                int h;
                if (a.draw) {
                    float sc[2];
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
                        const float* WT = hh ? WT1 : WT0;
                        const float* mu = hh ? mu1 : mu0;
                        float t[DV];
#pragma unroll
                        for (int l = 0; l < DV; ++l) t[l] = v[l] - mu[l];
                        float q = 0.f;
#pragma unroll
                        for (int j = 0; j < DV; ++j) {
                            if (j < d) {
                                float y = 0.f;
#pragma unroll
                                for (int l4 = 0; l4 <= j / 4; ++l4) {
                                    const float4 w = *(const float4*)(WT + j * DV + l4 * 4);
                                    y = fmaf(w.x, t[l4 * 4], y);
                                    y = fmaf(w.y, t[l4 * 4 + 1], y);
                                    y = fmaf(w.z, t[l4 * 4 + 2], y);
                                    y = fmaf(w.w, t[l4 * 4 + 3], y);
                                }
                                q = fmaf(y, y, q);
                            }
                        }
                        sc[hh] = cc[hh] - 0.5f * q;
                    }
                    uint32_t w[4];
                    key.block((uint32_t)i, TAG_ZBAR, 0, w);
                    const float vl = sc[0] + gumbel_of<float>(w[0], w[1]);
                    const float vr = sc[1] + gumbel_of<float>(w[2], w[3]);
                    h = vr > vl ? 1 : 0;
                    a.zbar[i] = (uint8_t)h;
                } else {
                    h = a.zbar[i];
                }
                // the centred row, then 1, then zeros, as float4 stores (conflict-free at any
                // row stride that is a multiple of 4 floats)
                float4* xr4 = (float4*)(xs + (size_t)tid * dp);
#pragma unroll
                for (int j4 = 0; j4 < (DV + 4) / 4; ++j4) {
                    if (j4 * 4 < dp) {
                        float e[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int j = 4 * j4 + u;
                            e[u] = j < d ? v[j < DV ? j : 0] - shf[j < DV ? j : 0] : (j == d ? 1.f : 0.f);
                        }
                        xr4[j4] = make_float4(e[0], e[1], e[2], e[3]);
                    }
                }
                hq[tid] = (unsigned char)h;
            }
        }
        __syncthreads();
        for (int r = 0; r < nr; ++r) {
            const int qs = runs[r], qe = runs[r + 1];
            const int k = kq[qs];
            if (k != cur) {
                if (cur >= 0) flush(cur);
                cur = k;
            }
            if (worker) {
                for (int q = qs + grp; q < qe; q += G) {
                    const float* xr = xs + (size_t)q * dp;
                    const float4 xj = *(const float4*)(xr + jb * 4);
                    const float4 xl = *(const float4*)(xr + lb * 4);
                    const float aj[4] = {xj.x, xj.y, xj.z, xj.w}, al[4] = {xl.x, xl.y, xl.z, xl.w};
                    if (hq[q]) {
#pragma unroll
                        for (int u = 0; u < 4; ++u)
#pragma unroll
                            for (int w2 = 0; w2 < 4; ++w2) acc1[u * 4 + w2] = fmaf(aj[u], al[w2], acc1[u * 4 + w2]);
                    } else {
#pragma unroll
                        for (int u = 0; u < 4; ++u)
#pragma unroll
                            for (int w2 = 0; w2 < 4; ++w2) acc0[u * 4 + w2] = fmaf(aj[u], al[w2], acc0[u * 4 + w2]);
                    }
                }
            }
        }
    }
    if (cur >= 0) flush(cur);
}

// FP32 variant for 64 < d <= 128 (Gaussian), two groups of warps.  The sorted positions of the
// block's range are cut into batches of at most WP = 64 points of one cluster.  The score
// group (8 warps) shifts batch i's rows by the cluster's centre, transposes them, and forms both
// Y_h = (X - shift) W_h - bh (bh = (mu_h - shift)^T W_h once per cluster) as register tiles of 8
// points x 4 columns, then the scores and z-bar; the statistics group (10 warps) adds batch i - 1
// to its register blocks (8 x 4 entries per thread and sub-cluster, every entry with one owner,
// written straight to the records); the rows of batch i + 1 arrive by cp.async meanwhile.
// What bounds it: shared-memory reads (12 floats a lane for 32 multiply-adds; LSU pipe 66% busy),
// then the FP32 FMA pipe.  W is upper triangular, so a tile of 16 columns ends at its last
// column's diagonal (56% of the square; a warp takes tiles i and 7 - i, 144 rows in all), and 14.3
// thousand FMA issues per scheduler and batch are left of 21.  Skipped products are exact zeros,
// every sum adds in the order l = 0, 1, ... (points: sorted order), and a score's 32 column
// groups are added by halves (16, 8, 4, 2, 1 apart).
// Measured at d = 128, N = 4e6, K = 64: 8.25 ms; 10.9 ms with square products and the two phases
// in turn over 18 warps.
// Dynamic shared memory: three row buffers of WP x dp, W_l and W_r as packed column tiles, the
// transposed rows (128 x TTS), the column groups' sums (2 x 32 x WP), then the small arrays.
constexpr int WP = 64;
constexpr int WIDE_S = 256;  // threads of the score group
constexpr int WIDE_T = 576;  // threads in all
constexpr int TTS = 68;      // row stride of the transposed rows
constexpr int WTILE = 16 * 16 * 36;  // floats of a packed factor: 8 column tiles of 16 (t + 1) rows

static size_t wide_smem_of(int dp) {
    return ((size_t)3 * WP * dp + 8 + 2 * WTILE + 128 * TTS + 64 * WP + 256 + 128 + 4) * 4 + (3 * WP + 260) * sizeof(int) + 3 * WP;
}

struct WideArgs {
    SubArgs<float> a;
    const int* starts;
};

__device__ __forceinline__ void wide_bar() { asm volatile("bar.sync 1, 256;" ::: "memory"); }  // the score group's

__global__ void __launch_bounds__(WIDE_T, 1) substats_wide_kernel(WideArgs wa) {
    const SubArgs<float>& a = wa.a;
    if (a.gate && *a.gate == 0) return;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int d = a.d, dp = a.L.dp, nb = a.L.nb;
    float* xs = (float*)smraw;                // 3 x WP x dp (+ 8: the last row's read past its end)
    float* Wp = xs + 3 * WP * dp + 8;         // 2 x WTILE
    float* Tt = Wp + 2 * WTILE;               // 128 x TTS
    float* qp = Tt + 128 * TTS;               // 2 x 32 x WP
    float* bh = qp + 64 * WP;                 // 2 x 128
    float* shf = bh + 256;                    // 128
    float* cc = shf + 128;                    // 2 (+ 2)
    int* iq = (int*)(cc + 4);                 // 3 x WP points
    int* st = iq + 3 * WP;                    // the range's clusters' starts
    unsigned char* hq = (unsigned char*)(st + 260);  // 3 x WP
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = blockIdx.x, K = *a.dK;
    const int64_t p0 = (int64_t)g * a.R, p1 = min(a.N, p0 + a.R);
    if (p0 >= p1 || K < 1) return;
    int k0 = 0;  // the cluster of position p0: the last k with starts[k] <= p0
    for (int lo = 0, hi = K; hi - lo > 1;) {
        const int mid = (lo + hi) >> 1;
        if (wa.starts[mid] <= p0) lo = mid;
        else hi = mid;
        k0 = lo;
    }
    // the batches, walked alike by every thread
    struct Batch {
        int64_t pos;
        int k, np, run;  // np = 0: none left; run: batch number
    };
    auto first_end = [&](int k) { return min(p1, (int64_t)(k - k0 < 259 ? st[k - k0 + 1] : wa.starts[k + 1])); };
    for (int e = tid; e < 260; e += WIDE_T) st[e] = k0 + e <= K ? wa.starts[k0 + e] : (int)min(a.N, (int64_t)0x7fffffff);
    __syncthreads();
    auto settle = [&](Batch& q) {  // q.pos, q.k -> the batch that begins there
        while (q.k + 1 < K && first_end(q.k) <= q.pos && q.pos < p1) ++q.k;
        q.np = q.pos < p1 ? (int)min((int64_t)WP, first_end(q.k) - q.pos) : 0;
        if (q.np < 0) q.np = 0;  // the starts do not cover the points (never for consistent state)
    };
    auto next = [&](Batch& q) {
        q.pos = q.np > 0 ? q.pos + q.np : p1;
        q.run += 1;
        settle(q);
    };
    Batch cur{p0, k0, 0, 0};
    settle(cur);

    if (warp < WIDE_S / 32) {
        // ------------------------------------------------------------ score group
        const Key key{a.seed, a.diter[0], a.diter[1], a.diter[2]};
        const float* X = (const float*)a.X;
        // rows 8 warp .. 8 warp + 7 of a batch: lane r < 8 holds row r's point
        auto load_idx = [&](const Batch& q) {
            const int r = 8 * warp + lane;
            return lane < 8 && r < q.np ? a.idx[q.pos + r] : 0;
        };
        auto fetch = [&](const Batch& q, int pt) {
            float* to = xs + (size_t)(q.run % 3) * WP * dp;
            for (int r = 0; r < 8; ++r) {
                const int i = __shfl_sync(0xffffffffu, pt, r), row = 8 * warp + r;
                if (row < q.np && lane * 4 < d) mw_cp16(to + row * dp + lane * 4, X + (int64_t)i * a.xs + lane * 4);
            }
            if (lane < 8) iq[(q.run % 3) * WP + 8 * warp + lane] = pt;
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        Batch nx = cur;
        fetch(cur, load_idx(cur));
        next(nx);
        int pt = load_idx(nx);
        int staged = -1;
        for (; cur.np > 0;) {
            Batch n2 = nx;
            if (nx.np > 0) {
                fetch(nx, pt);
                next(n2);
                pt = load_idx(n2);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            const int np = cur.np, k = cur.k, buf = cur.run % 3;
            float* xb = xs + (size_t)buf * WP * dp;
            if (k != staged) {  // the cluster's two sub-clusters (every reader of the last is past a barrier)
                for (int e = tid; e < 2 * WTILE; e += WIDE_S) {
                    const int h = e / WTILE, f = e % WTILE, r16 = f >> 4;  // 16-float row r16 of the packed tiles
                    int t = 0;
                    while (8 * (t + 1) * (t + 2) <= r16) ++t;
                    const int l = r16 - 8 * t * (t + 1), j = 16 * t + (f & 15);
                    Wp[e] = (j < d && l <= j) ? a.pv.W[((size_t)(3 * k + 1 + h) * d + l) * d + j] : 0.f;
                }
                if (tid < 2) cc[tid] = a.pv.c[3 * k + 1 + tid];
                if (tid < 128) shf[tid] = tid < d ? a.shift[(size_t)k * d + tid] : 0.f;
                wide_bar();
                {  // bh[h][j] = sum_l (mu_h - shift)_l W_h[l][j]
                    const int h = tid >> 7, j = tid & 127, t = j >> 4;
                    const float* mu = a.pv.mu + (size_t)(3 * k + 1 + h) * d;
                    const float* Wt = Wp + h * WTILE + 128 * t * (t + 1) + (j & 15);
                    float b = 0.f;
                    if (j < d)
                        for (int l = 0; l <= j; ++l) b = fmaf(__ldg(mu + l) - shf[l], Wt[l * 16], b);
                    bh[tid] = b;
                }
                staged = k;
            }
            wide_bar();  // the rows have landed, the parameters are staged
            // the rows less the centre, then 1, then zeros; and transposed
            for (int p = warp; p < WP; p += WIDE_S / 32) {
                float* xr = xb + p * dp;
                for (int j = lane; j < max(dp, 128); j += 32) {
                    float v = 0.f;
                    if (p < np) v = j < d ? xr[j] - shf[j] : (j == d ? 1.f : 0.f);
                    if (j < dp) xr[j] = v;
                    if (j < 128) Tt[j * TTS + p] = j < d ? v : 0.f;
                }
            }
            if (a.draw) {
                wide_bar();
                const int h = warp >> 2, pg = lane & 7, cg = lane >> 3;  // points 8 pg .., columns 16 t + 4 cg ..
                for (int half = 0; half < 2; ++half) {
                    const int t = half ? warp & 3 : 7 - (warp & 3);
                    if (16 * t >= d) {  // no such columns: zero sums, as their products would give
                        for (int u = 0; u < 8; ++u) qp[(h * 32 + 4 * t + cg) * WP + 8 * pg + u] = 0.f;
                        continue;
                    }
                    float y[8][4];
#pragma unroll
                    for (int u = 0; u < 8; ++u)
#pragma unroll
                        for (int v = 0; v < 4; ++v) y[u][v] = 0.f;
                    const float* Wt = Wp + h * WTILE + 128 * t * (t + 1) + 4 * cg;
                    const float* tp = Tt + 8 * pg;
                    const int le = min(d, 16 * t + 16);
#pragma unroll 4
                    for (int l = 0; l < le; ++l) {
                        const float4 t0 = *(const float4*)(tp + l * TTS);
                        const float4 t1 = *(const float4*)(tp + l * TTS + 4);
                        const float4 w0 = *(const float4*)(Wt + l * 16);
                        const float tv[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
                        const float wv[4] = {w0.x, w0.y, w0.z, w0.w};
#pragma unroll
                        for (int u = 0; u < 8; ++u)
#pragma unroll
                            for (int v = 0; v < 4; ++v) y[u][v] = fmaf(tv[u], wv[v], y[u][v]);
                    }
                    const float4 b4 = *(const float4*)(bh + h * 128 + 16 * t + 4 * cg);
                    const float bv[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        float s0 = 0.f;
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            const float r = y[u][v] - bv[v];
                            s0 = fmaf(r, r, s0);
                        }
                        qp[(h * 32 + 4 * t + cg) * WP + 8 * pg + u] = s0;
                    }
                }
                wide_bar();
            }
            if (tid < np) {
                const int i = iq[buf * WP + tid];
                int h;
                if (a.draw) {
                    float q[2];
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {  // the column groups 16, 8, 4, 2, 1 apart
                        float v[16];
#pragma unroll
                        for (int c = 0; c < 16; ++c) v[c] = qp[(hh * 32 + c) * WP + tid] + qp[(hh * 32 + c + 16) * WP + tid];
#pragma unroll
                        for (int o = 8; o > 0; o >>= 1)
#pragma unroll
                            for (int c = 0; c < o; ++c) v[c] += v[c + o];
                        q[hh] = v[0];
                    }
                    uint32_t w[4];
                    key.block((uint32_t)i, TAG_ZBAR, 0, w);
                    const float vl = cc[0] - 0.5f * q[0] + gumbel_of<float>(w[0], w[1]);
                    const float vr = cc[1] - 0.5f * q[1] + gumbel_of<float>(w[2], w[3]);
                    h = vr > vl ? 1 : 0;
                    a.zbar[i] = (uint8_t)h;
                } else {
                    h = a.zbar[i];
                }
                hq[buf * WP + tid] = (unsigned char)h;
            }
            __syncthreads();  // batch cur is ready for the statistics group, batch cur - 1 added up
            cur = nx;
            nx = n2;
        }
        __syncthreads();  // the last batch added up
    } else {
        // ------------------------------------------------------------ statistics group
        const int t = tid - WIDE_S;
        int J = 0, lb = t;  // rows 8 J .. 8 J + 7, columns 4 lb .. 4 lb + 3 (blocks 2 J <= lb, 2 J + 1 <= lb)
        bool worker = true;
        while (worker && lb >= nb - 2 * J) {
            lb -= nb - 2 * J;
            ++J;
            worker = 2 * J < nb;
        }
        lb += 2 * J;
        float acc0[32], acc1[32];
#pragma unroll
        for (int e = 0; e < 32; ++e) acc0[e] = acc1[e] = 0.f;
        auto flush = [&](int k) {
            if (worker) {
                double* out = a.rec + (size_t)(g + k) * 2 * a.L.E;
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    const int jb = 2 * J + v;
                    if (jb > lb || jb >= nb) continue;
                    double* o = out + (size_t)a.L.blk(jb, lb) * 16;
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        o[e] = (double)acc0[16 * v + e];
                        o[a.L.E + e] = (double)acc1[16 * v + e];
                    }
                }
            }
#pragma unroll
            for (int e = 0; e < 32; ++e) acc0[e] = acc1[e] = 0.f;
        };
        Batch prev = cur;
        for (bool more = cur.np > 0; more;) {
            __syncthreads();  // batch prev is ready
            next(cur);
            more = cur.np > 0;
            const float* xb = xs + (size_t)(prev.run % 3) * WP * dp;
            const unsigned char* hb = hq + (prev.run % 3) * WP;
            if (worker) {
                for (int q = 0; q < prev.np; ++q) {
                    const float* xr = xb + q * dp;
                    const float4 j0 = *(const float4*)(xr + J * 8), j1 = *(const float4*)(xr + J * 8 + 4);
                    const float4 xl = *(const float4*)(xr + lb * 4);
                    const float aj[8] = {j0.x, j0.y, j0.z, j0.w, j1.x, j1.y, j1.z, j1.w}, al[4] = {xl.x, xl.y, xl.z, xl.w};
                    if (hb[q]) {
#pragma unroll
                        for (int u = 0; u < 8; ++u)
#pragma unroll
                            for (int v = 0; v < 4; ++v) acc1[u * 4 + v] = fmaf(aj[u], al[v], acc1[u * 4 + v]);
                    } else {
#pragma unroll
                        for (int u = 0; u < 8; ++u)
#pragma unroll
                            for (int v = 0; v < 4; ++v) acc0[u * 4 + v] = fmaf(aj[u], al[v], acc0[u * 4 + v]);
                    }
                }
            }
            if (!more || cur.k != prev.k) flush(prev.k);
            prev = cur;
        }
        __syncthreads();
    }
}

// Multinomial variant (first-moment statistics only): the point's counts become a
// float row in shared memory (x, then 1, then zeros), each row loaded by one warp in
// 16-byte pieces, four rows in flight per lane; the current run's two sub-cluster log
// theta vectors are staged in shared memory; each sub-cluster score is a d-long dot
// product fed by float4 loads; each worker thread owns the counts of one 4-category
// block for both sub-clusters.  Dynamic shared memory: P x dp rows, P ints (k), P + 2
// ints (runs), P ints (point indices), P bytes (h), then 2 dp + 2 floats (staged
// parameters), then the flush buffer G x nblk x 8 floats.
template <typename XT>
__global__ void __launch_bounds__(256) substats_mult_kernel(SubArgs<float> a) {
    if (a.gate && *a.gate == 0) return;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int d = a.d, dp = a.L.dp, P = a.P, G = a.G, nblk = a.L.nblk;
    float* xs = (float*)smraw;
    int* kq = (int*)(xs + (size_t)P * dp);
    int* runs = kq + P;
    int* nruns = runs + P + 1;
    int* iq = nruns + 1;
    unsigned char* hq = (unsigned char*)(iq + P);
    float* lt0 = (float*)(smraw + (((size_t)P * dp * 4 + (3 * P + 2) * sizeof(int) + P + 15) / 16) * 16);
    float* lt1 = lt0 + dp;
    float* cc = lt1 + dp;
    float* red = (float*)(((uintptr_t)(cc + 2) + 15) & ~(uintptr_t)15);
    __shared__ int staged;
    __shared__ int wcnt[32];

    const int tid = threadIdx.x, nt = blockDim.x;
    const int g = blockIdx.x;
    const int64_t p0 = (int64_t)g * a.R, p1 = min(a.N, p0 + a.R);
    Key key{a.seed, a.diter[0], a.diter[1], a.diter[2]};
    const XT* X = (const XT*)a.X;
    const bool worker = tid < nblk * G;
    const int myblk = worker ? tid % nblk : 0, grp = worker ? tid / nblk : 0;
    const int one = d & 3;  // position of the constant 1 inside the last 4-column block
    float acc0[4] = {0.f, 0.f, 0.f, 0.f}, acc1[4] = {0.f, 0.f, 0.f, 0.f};
    int cur = -1;
    if (tid == 0) staged = -1;

    auto flush = [&](int k) {
        __syncthreads();
        if (worker) {
            float* r = red + ((size_t)grp * nblk + myblk) * 8;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                r[u] = acc0[u];
                r[4 + u] = acc1[u];
            }
        }
        __syncthreads();
        double* out = a.rec + (size_t)(g + k) * 2 * a.L.E;
        for (int e = tid; e < nblk * 16; e += nt) {
            const int b = e >> 4, q = e & 15, u = q >> 2, v = q & 3;
            double s0 = 0.0, s1 = 0.0;
            if (v == one)
                for (int gg = 0; gg < G; ++gg) {
                    s0 += (double)red[((size_t)gg * nblk + b) * 8 + u];
                    s1 += (double)red[((size_t)gg * nblk + b) * 8 + 4 + u];
                }
            out[e] = s0;
            out[a.L.E + e] = s1;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) acc0[u] = acc1[u] = 0.f;
    };

    for (int64_t base = p0; base < p1; base += P) {
        const int np = (int)min((int64_t)P, p1 - base);
        __syncthreads();
        int i = 0;
        if (tid < np) {
            i = a.idx[base + tid];
            kq[tid] = a.z[i];
            iq[tid] = i;
        }
        __syncthreads();
        {
            const int lane = tid & 31, nwarp = nt >> 5;
            if constexpr (sizeof(XT) == 2) {  // 16-byte loads: 8 BF16 counts (rows are 16-byte aligned)
                const int nfull = d / 8;      // whole 8-count chunks inside the row's d columns
                for (int q0 = tid >> 5; q0 < np; q0 += 4 * nwarp) {
                    for (int c0 = 0; c0 < nfull; c0 += 32) {
                        const int c8 = c0 + lane;
                        uint4 v[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int q = q0 + u * nwarp;
                            if (q < np && c8 < nfull) v[u] = ((const uint4*)(X + (int64_t)iq[q] * a.xs))[c8];
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int q = q0 + u * nwarp;
                            if (q < np && c8 < nfull) {
                                const uint32_t wv[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
                                float f[8];
#pragma unroll
                                for (int w = 0; w < 4; ++w) {
                                    f[2 * w] = __uint_as_float(wv[w] << 16);
                                    f[2 * w + 1] = __uint_as_float(wv[w] & 0xFFFF0000u);
                                }
                                float* xr = xs + (size_t)q * dp + 8 * c8;
                                *(float4*)xr = make_float4(f[0], f[1], f[2], f[3]);
                                *(float4*)(xr + 4) = make_float4(f[4], f[5], f[6], f[7]);
                            }
                        }
                    }
                    for (int u = 0; u < 4; ++u) {
                        const int q = q0 + u * nwarp;
                        if (q >= np) break;
                        for (int j = 8 * nfull + lane; j < dp; j += 32)
                            xs[(size_t)q * dp + j] = j < d ? ldx<float, XT>(X + (int64_t)iq[q] * a.xs + j) : (j == d ? 1.f : 0.f);
                    }
                }
            } else {
                for (int q = tid >> 5; q < np; q += nwarp)
                    for (int j = lane; j < dp; j += 32)
                        xs[(size_t)q * dp + j] = j < d ? ldx<float, XT>(X + (int64_t)iq[q] * a.xs + j) : (j == d ? 1.f : 0.f);
            }
        }
        __syncthreads();
        find_runs(kq, np, runs, nruns, wcnt);
        const int nr = *nruns;
        for (int r = 0; r < nr; ++r) {
            const int qs = runs[r], qe = runs[r + 1];
            const int k = kq[qs];
            if (a.draw && k != staged) {  // uniform: stage this cluster's two sub-clusters
                __syncthreads();
                for (int e = tid; e < 2 * dp; e += nt) {
                    const int h = e / dp, j = e % dp;
                    lt0[e] = j < d ? a.pv.lt[(size_t)(3 * k + 1 + h) * d + j] : 0.f;
                }
                if (tid < 2) cc[tid] = a.pv.c[3 * k + 1 + tid];
                __syncthreads();
                if (tid == 0) staged = k;
            }
            if (tid >= qs && tid < qe) {
                int h;
                if (a.draw) {
                    const float4* xr4 = (const float4*)(xs + (size_t)tid * dp);
                    const float4* l04 = (const float4*)lt0;
                    const float4* l14 = (const float4*)lt1;
                    float s0 = 0.f, s1 = 0.f, t0 = 0.f, t1 = 0.f;
                    for (int j4 = 0; j4 < dp / 4; ++j4) {
                        const float4 x = xr4[j4], u = l04[j4], w = l14[j4];
                        s0 = fmaf(x.x, u.x, s0);
                        t0 = fmaf(x.y, u.y, t0);
                        s0 = fmaf(x.z, u.z, s0);
                        t0 = fmaf(x.w, u.w, t0);
                        s1 = fmaf(x.x, w.x, s1);
                        t1 = fmaf(x.y, w.y, t1);
                        s1 = fmaf(x.z, w.z, s1);
                        t1 = fmaf(x.w, w.w, t1);
                    }
                    // the padding column d holds 1 and lt[d] = 0: it adds nothing
                    uint32_t wq[4];
                    key.block((uint32_t)i, TAG_ZBAR, 0, wq);
                    const float vl = cc[0] + s0 + t0 + gumbel_of<float>(wq[0], wq[1]);
                    const float vr = cc[1] + s1 + t1 + gumbel_of<float>(wq[2], wq[3]);
                    h = vr > vl ? 1 : 0;
                    a.zbar[i] = (uint8_t)h;
                } else {
                    h = a.zbar[i];
                }
                hq[tid] = (unsigned char)h;
            }
        }
        __syncthreads();
        for (int r = 0; r < nr; ++r) {
            const int qs = runs[r], qe = runs[r + 1];
            const int k = kq[qs];
            if (k != cur) {
                if (cur >= 0) flush(cur);
                cur = k;
            }
            if (worker) {
                for (int q = qs + grp; q < qe; q += G) {
                    const float4 xj = *(const float4*)(xs + (size_t)q * dp + myblk * 4);
                    if (hq[q]) {
                        acc1[0] += xj.x; acc1[1] += xj.y; acc1[2] += xj.z; acc1[3] += xj.w;
                    } else {
                        acc0[0] += xj.x; acc0[1] += xj.y; acc0[2] += xj.z; acc0[3] += xj.w;
                    }
                }
            }
        }
    }
    if (cur >= 0) flush(cur);
}

// Multinomial sub-labels and statistics (first moments only), one warp per range of sorted
// positions, that is, of points in cluster order.  Lane l holds categories 8l .. 8l + 7 (d <= 256)
// of a point's counts and of the two sub-cluster log theta rows of the current cluster; the
// two sub-cluster scores are dot products reduced across the warp; the z-bar draws of 32
// points are made at once, one point per lane, and four points' scores are reduced together
// (N = 1e6, d = 200, K = 50: 187 us, from 238 us with two five-step reductions a point).  The
// counts of a cluster's run stay in registers and are added at the run's end to the compact table cnt (2 K_max x (d + 1) integers, column
// d: the points) with atomic adds, exact in any order.  No block-wide barrier.
struct MwArgs {
    int64_t N, R;  // points; sorted positions per warp
    int d, xs;
    const void* X;
    const int* idx;     // sorted position -> point
    const int* starts;  // K + 1 cluster offsets in sorted order
    const int* dK;
    const float* lt;    // slots x d log theta (FP32)
    const float* lc;    // slots: log weights
    const uint32_t* diter;
    uint64_t seed;
    const int* gate;
    int draw;
    uint8_t* zbar;
    unsigned* cnt;
};

constexpr int MW_DEPTH = 16;  // rows in flight per warp (a ring in shared memory)
constexpr int MW_ROWB = 512;  // bytes per ring slot: d <= 256 BF16 counts

// BF16 counts (rows 16-byte aligned).  Dynamic shared memory: 8 warps x MW_DEPTH x MW_ROWB.
__global__ void __launch_bounds__(256, 3) mult_warp_kernel(MwArgs a) {
    if (a.gate && *a.gate == 0) return;
    extern __shared__ __align__(16) unsigned char mw_sm[];
    const int lane = threadIdx.x & 31;
    unsigned char* ring = mw_sm + (threadIdx.x >> 5) * (MW_DEPTH * MW_ROWB);
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t p0 = w * a.R, p1 = min(a.N, p0 + a.R);
    if (p0 >= p1) return;
    const int K = *a.dK, d = a.d, j0 = 8 * lane, nch = (d + 7) >> 3;
    int k = 0;  // the cluster of position p0: the last k with starts[k] <= p0
    for (int lo = 0, hi = K; hi - lo > 1;) {
        const int mid = (lo + hi) >> 1;
        if (a.starts[mid] <= p0) lo = mid;
        else hi = mid;
        k = lo;
    }
    int64_t kend = a.starts[k + 1];
    float lt0[8], lt1[8], c0 = 0.f, c1 = 0.f;
    auto stage = [&](int kk) {
        const float* r0 = a.lt + (size_t)(3 * kk + 1) * d + j0;
        const float* r1 = r0 + d;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            lt0[u] = j0 + u < d ? r0[u] : 0.f;
            lt1[u] = j0 + u < d ? r1[u] : 0.f;
        }
        c0 = a.lc[3 * kk + 1];
        c1 = a.lc[3 * kk + 2];
    };
    unsigned acc0[8], acc1[8], n0 = 0, n1 = 0;  // integer counts: exact
#pragma unroll
    for (int u = 0; u < 8; ++u) acc0[u] = acc1[u] = 0u;
    auto flush = [&](int kk) {
        unsigned* r0 = a.cnt + (size_t)(2 * kk) * (d + 1);
        unsigned* r1 = r0 + (d + 1);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (j0 + u < d) {
                if (acc0[u]) atomicAdd(r0 + j0 + u, acc0[u]);
                if (acc1[u]) atomicAdd(r1 + j0 + u, acc1[u]);
            }
            acc0[u] = acc1[u] = 0u;
        }
        if (lane == 0) {
            if (n0) atomicAdd(r0 + d, n0);
            if (n1) atomicAdd(r1 + d, n1);
        }
        n0 = n1 = 0;
    };
    if (a.draw) stage(k);
    const Key key{a.seed, a.diter[0], a.diter[1], a.diter[2]};
    // point indices of positions in batches of 32 (lane l: position batch start + l); the
    // next batch's are loaded one batch ahead
    int64_t bstart = p0;
    int cur = p0 + lane < p1 ? a.idx[p0 + lane] : 0;
    int nxt = p0 + 32 + lane < p1 ? a.idx[p0 + 32 + lane] : 0;
    auto pick = [&](int64_t pos) {
        const int r = (int)(pos - bstart);
        const int vc = __shfl_sync(0xffffffffu, cur, r & 31), vn = __shfl_sync(0xffffffffu, nxt, r & 31);
        return r < 32 ? vc : vn;
    };
    auto issue = [&](int slot, int64_t pos) {  // the row of position pos into a ring slot
        if (pos < p1) {
            const int i = pick(pos);
            if (lane < nch)
                mw_cp16(ring + slot * MW_ROWB + lane * 16, (const char*)a.X + (int64_t)i * a.xs * 2 + lane * 16);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int t = 0; t < MW_DEPTH; ++t) issue(t, p0 + t);
    float gl = 0.f, gr = 0.f;
    int hz = 0;
    auto draws = [&]() {  // this batch's z-bar Gumbel values (or kept z-bar), one point per lane
        if (bstart + lane < p1) {
            if (a.draw) {
                uint32_t wq[4];
                key.block((uint32_t)cur, TAG_ZBAR, 0, wq);
                gl = gumbel_of<float>(wq[0], wq[1]);
                gr = gumbel_of<float>(wq[2], wq[3]);
            } else {
                hz = a.zbar[cur];
            }
        }
    };
    draws();
    auto unpack = [](const uint4& q, float* x) {  // the row's padding beyond d is zero
        const uint32_t wv[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            x[2 * u] = __uint_as_float(wv[u] << 16);
            x[2 * u + 1] = __uint_as_float(wv[u] & 0xFFFF0000u);
        }
    };
    auto add = [&](const uint4& q, int h) {
        float x[8];
        unpack(q, x);
        if (h) {
#pragma unroll
            for (int u = 0; u < 8; ++u) acc1[u] += (unsigned)x[u];
            ++n1;
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) acc0[u] += (unsigned)x[u];
            ++n0;
        }
    };
    for (int64_t p = p0; p < p1; p += 4) {  // four points at a time
        if (p - bstart == 32) {  // the next batch
            bstart += 32;
            cur = nxt;
            nxt = bstart + 32 + lane < p1 ? a.idx[bstart + 32 + lane] : 0;
            draws();
        }
        const int slot = (int)((p - p0) % MW_DEPTH);
        asm volatile("cp.async.wait_group %0;" ::"n"(MW_DEPTH - 4) : "memory");
        __syncwarp();
        uint4 row[4];  // unpacked where used: the registers hold two rows of floats at most
#pragma unroll
        for (int v = 0; v < 4; ++v)
            row[v] = lane < nch ? *(const uint4*)(ring + (slot + v) * MW_ROWB + lane * 16) : make_uint4(0u, 0u, 0u, 0u);
        __syncwarp();  // every lane has read the slots: they may be refilled
#pragma unroll
        for (int v = 0; v < 4; ++v) issue(slot + v, p + MW_DEPTH + v);
        const int q = (int)(p - bstart);
        if (a.draw && p + 4 <= min(p1, kend)) {
            // Eight sums (two scores of four points) reduced across the lanes at once: at each
            // of the first three levels a lane keeps one of two values and hands the other over,
            // so 9 exchanges do the work of 40; every sum adds lanes 16, 8, 4, 2, 1 apart, in
            // that order, as reducing each on its own would.
            float t[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                float s0 = 0.f, s1 = 0.f, x[8];
                unpack(row[v], x);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    s0 = fmaf(x[u], lt0[u], s0);
                    s1 = fmaf(x[u], lt1[u], s1);
                }
                const bool up = lane & 16;
                t[v] = (up ? s1 : s0) + __shfl_xor_sync(0xffffffffu, up ? s0 : s1, 16);
            }
            const bool b8 = lane & 8, b4 = lane & 4;
            const float m0 = (b8 ? t[1] : t[0]) + __shfl_xor_sync(0xffffffffu, b8 ? t[0] : t[1], 8);
            const float m1 = (b8 ? t[3] : t[2]) + __shfl_xor_sync(0xffffffffu, b8 ? t[2] : t[3], 8);
            float w = (b4 ? m1 : m0) + __shfl_xor_sync(0xffffffffu, b4 ? m0 : m1, 4);
            w += __shfl_xor_sync(0xffffffffu, w, 2);
            w += __shfl_xor_sync(0xffffffffu, w, 1);
            // lane bits 16: sub-cluster, 8 and 4: point
            const int pt = (b4 ? 2 : 0) + (b8 ? 1 : 0);
            const float el = __shfl_sync(0xffffffffu, gl, q + pt), er = __shfl_sync(0xffffffffu, gr, q + pt);
            const float val = (lane & 16 ? c1 : c0) + w + (lane & 16 ? er : el);
            const float oth = __shfl_xor_sync(0xffffffffu, val, 16);
            const unsigned m = __ballot_sync(0xffffffffu, oth > val);  // lanes 0, 8, 4, 12: points 0 .. 3
            const int h[4] = {(int)(m & 1u), (int)(m >> 8 & 1u), (int)(m >> 4 & 1u), (int)(m >> 12 & 1u)};
            const int r = lane - q;
            if (r >= 0 && r < 4) a.zbar[cur] = (uint8_t)(r == 0 ? h[0] : r == 1 ? h[1] : r == 2 ? h[2] : h[3]);
#pragma unroll
            for (int v = 0; v < 4; ++v) add(row[v], h[v]);
            continue;
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            if (p + v >= p1) break;
            while (p + v >= kend) {  // the next cluster's run begins
                flush(k);
                ++k;
                kend = a.starts[k + 1];
                if (a.draw) stage(k);
            }
            int h;
            if (a.draw) {
                float s0 = 0.f, s1 = 0.f, x[8];
                unpack(row[v], x);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    s0 = fmaf(x[u], lt0[u], s0);
                    s1 = fmaf(x[u], lt1[u], s1);
                }
                for (int o = 16; o > 0; o >>= 1) {
                    s0 += __shfl_xor_sync(0xffffffffu, s0, o);
                    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
                }
                const float vl = c0 + s0 + __shfl_sync(0xffffffffu, gl, q + v);
                const float vr = c1 + s1 + __shfl_sync(0xffffffffu, gr, q + v);
                h = vr > vl ? 1 : 0;
                if (lane == q + v) a.zbar[cur] = (uint8_t)h;
            } else {
                h = __shfl_sync(0xffffffffu, hz, q + v);
            }
            add(row[v], h);
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    flush(k);
}

// the compact counts of the 2K sub-clusters: cleared before, copied into the FP64
// statistics table after (grid: y = sub-cluster slot, x strides over the d + 1 columns)
__global__ void mcnt_zero_kernel(const int* dK, const int* gate, int d, unsigned* cnt) {
    if (gate && *gate == 0) return;
    const int s = blockIdx.y;
    if (s >= 2 * *dK) return;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j <= d; j += gridDim.x * blockDim.x) cnt[(size_t)s * (d + 1) + j] = 0u;
}

__global__ void mcnt_fill_kernel(const int* dK, const int* gate, StatLayout L, const unsigned* cnt, double* S) {
    if (gate && *gate == 0) return;
    const int s = blockIdx.y, d = L.d;
    if (s >= 2 * *dK) return;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j <= d; j += gridDim.x * blockDim.x)
        S[(size_t)s * L.E + L.ent(j, d)] = (double)cnt[(size_t)s * (d + 1) + j];
}

// stats[(2k + h) E + e] = sum over the CTAs g covering cluster k's run of rec[g + k]
__global__ void combine_kernel(const double* rec, const int* starts, const int* dK, int64_t R, int E,
                               const double* shift_new, double* shift_stats, int d, const int* gate,
                               double* stats) {
    if (gate && *gate == 0) return;
    const int K = *dK;
    const int kh = blockIdx.y, k = kh >> 1, h = kh & 1;
    if (k >= K) return;
    const int64_t st = starts[k], cnt = (int64_t)starts[k + 1] - st;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (blockIdx.x == 0 && h == 0)
        for (int j = threadIdx.x; j < d; j += blockDim.x) shift_stats[(size_t)k * d + j] = shift_new[(size_t)k * d + j];
    if (e >= E) return;
    double v = 0.0;
    if (cnt > 0) {  // the ranges' records in order; four loads in flight at a time
        const int64_t g0 = st / R, g1 = (st + cnt - 1) / R;
        for (int64_t g = g0; g <= g1; g += 4) {
            double r[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) r[u] = g + u <= g1 ? rec[((size_t)(g + u + k) * 2 + h) * E + e] : 0.0;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (g + u <= g1) v += r[u];
        }
    }
    stats[(size_t)kh * E + e] = v;
}

// initial labels: K = init_K, z uniform over K, z-bar a fair coin (tag INIT, c1 = 0)
__global__ void init_labels_kernel(int64_t N, int initK, uint64_t seed, const uint32_t* diter, int32_t* z,
                                   uint8_t* zbar) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    Key key{seed, 0, diter[1], diter[2]};
    uint32_t w[4];
    key.block((uint32_t)i, TAG_INIT, 0, w);
    int k = (int)(u01_f64(w[0], w[1]) * initK);
    if (k >= initK) k = initK - 1;
    z[i] = k;
    zbar[i] = u01_f64(w[2], w[3]) < 0.5 ? 0 : 1;
}

// ------------------------------------------------------------------ launchers
template <typename T>
static ParamView<T> pview(dpmm_ctx* c);
template <>
ParamView<double> pview<double>(dpmm_ctx* c) { return {c->p_W, c->p_mu, c->p_c, c->p_logtheta}; }
template <>
ParamView<float> pview<float>(dpmm_ctx* c) { return {c->q_W, c->q_mu, c->q_c, c->q_logtheta}; }

template <typename T, typename XT>
static cudaError_t labels_simt_t(dpmm_ctx* c, uint64_t seed, const int* gate) {
    const int d = c->d;
    const size_t per = c->kind == DPMM_PRIOR_NIW ? (size_t)d * d + d + 1 : (size_t)d + 1;
    size_t budget = 200 * 1024;
    int TB = 256;  // fewer points per CTA when the rows would not leave room for one cluster
    while (TB > 32 && (size_t)TB * (d + 1) * sizeof(T) + per * sizeof(T) > budget / 2) TB /= 2;
    const size_t rows = (size_t)TB * (d + 1) * sizeof(T);
    if (rows + per * sizeof(T) > budget) return cudaErrorInvalidValue;  // d too large for this kernel
    int CB = (int)std::max<size_t>(1, std::min<size_t>(32, (budget - rows) / (per * sizeof(T))));
    size_t sm = CB * per * sizeof(T) + rows;
    auto kern = c->dbg_scores ? labels_simt_kernel<T, XT, true> : labels_simt_kernel<T, XT, false>;
    cudaError_t ea = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (ea != cudaSuccess) return ea;
    // a gated launch usually exits at once: one wave of CTAs (one per SM at this shared
    // memory size) that stride over the tiles
    int64_t tiles = (c->N + TB - 1) / TB;
    int grid = (int)(gate ? std::min<int64_t>(tiles, (int64_t)c->num_sms) : tiles);
    kern<<<grid, TB, sm, c->stream>>>(c->kind, d, c->xs, c->N, (const XT*)c->X, pview<T>(c), c->dK, c->diter, seed,
                                      CB, gate, c->dbg_scores, c->z);
    return cudaGetLastError();
}

// Gaussian FP64 labels without the score hook.  Blocks of 32 to 128 points: the most that
// still give every SM two blocks.
static cudaError_t labels_niw64(dpmm_ctx* c, uint64_t seed) {
    const int d = c->d;
    const size_t per = ((size_t)d * d + d + 1) * sizeof(double);  // d too large for labels_simt_kernel: refused here too
    if ((size_t)32 * (d + 1) * sizeof(double) + per > 200 * 1024) return cudaErrorInvalidValue;
    const size_t stg = (((NIW_B + 1) * (size_t)d + 3) & ~(size_t)3) * 2 * 4;  // per warp
    auto bytes = [&](int TB) { return (size_t)d * (TB + 1) * 16 + 16 + (size_t)NIW_C * TB * 16 + (size_t)NIW_P * TB * 2 + (size_t)(TB / 32) * stg; };
    int TB = 128;
    while (TB > 32 && (bytes(TB) > 100 * 1024 || c->N < (int64_t)TB * 2 * c->num_sms)) TB /= 2;
    auto kern = d % 4 == 0 ? labels_niw64_kernel<true> : labels_niw64_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes(TB));
    if (e != cudaSuccess) return e;
    const int grid = (int)((c->N + TB - 1) / TB);
    Niw64 a{d, c->xs, c->N, (const double*)c->X, c->p_W, c->p_mu, c->p_c, c->q_W, c->q_mu, c->q_b,
            c->q_c, c->sorted ? c->idx : nullptr, c->dK, c->diter, seed, c->z};
    kern<<<grid, TB, bytes(TB), c->stream>>>(a);
    return cudaGetLastError();
}

// labels_small_kernel where it applies: the padded parameters of K_max clusters in 100 KB, two blocks to
// an SM (the launch does not know K).  Beyond (FP32: K_max 93 at d > 8, 350 at d > 4; FP64: 175 at
// d > 4) the kernels of larger d take over, which stage clusters in turn.
template <typename T, int DV>
static cudaError_t labels_small_t(dpmm_ctx* c, uint64_t seed) {
    const size_t smem = (size_t)c->K_max * (DV * DV + DV + 1) * sizeof(T);
    const int64_t room = 2048 * (int64_t)c->num_sms;  // resident threads
    const int L = c->N * 8 <= room ? 8 : c->N * 4 <= room ? 4 : c->N * 2 <= room ? 2 : 1;
    auto kern = L == 8 ? labels_small_kernel<T, DV, 8> : L == 4 ? labels_small_kernel<T, DV, 4>
              : L == 2 ? labels_small_kernel<T, DV, 2> : labels_small_kernel<T, DV, 1>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int64_t blocks = (c->N * L + 255) / 256;
    kern<<<(int)std::min<int64_t>(blocks, 8 * (int64_t)c->num_sms), 256, smem, c->stream>>>(
        c->d, c->xs, c->N, (const T*)c->X, pview<T>(c), c->dK, c->diter, seed, c->z);
    return cudaGetLastError();
}

static bool labels_small(const dpmm_ctx* c) {
    const bool f64 = c->prec == DPMM_PREC_FP64_PLAIN;
    const int DV = c->d <= 2 ? 2 : c->d <= 4 ? 4 : c->d <= 8 ? 8 : 16;
    return c->kind == DPMM_PRIOR_NIW && c->d <= (f64 ? 8 : 16) && !c->dbg_scores &&
           (size_t)c->K_max * (DV * DV + DV + 1) * (f64 ? 8 : 4) <= 100 * 1024;
}

cudaError_t launch_labels_simt_gated(dpmm_ctx* c, uint64_t seed, const int* gate) {
    const char* name = gate ? "labels_simt_overflow" : "labels_simt";
    prof_begin(c, name);
    cudaError_t e;
    if (!gate && labels_small(c)) {
        if (c->prec == DPMM_PREC_FP64_PLAIN)
            e = c->d <= 2 ? labels_small_t<double, 2>(c, seed) : c->d <= 4 ? labels_small_t<double, 4>(c, seed)
                                                               : labels_small_t<double, 8>(c, seed);
        else
            e = c->d <= 2 ? labels_small_t<float, 2>(c, seed) : c->d <= 4 ? labels_small_t<float, 4>(c, seed)
              : c->d <= 8 ? labels_small_t<float, 8>(c, seed) : labels_small_t<float, 16>(c, seed);
    } else if (c->kind == DPMM_PRIOR_NIW && c->prec == DPMM_PREC_FP64_PLAIN && !c->dbg_scores) e = labels_niw64(c, seed);
    else if (c->prec == DPMM_PREC_FP64_PLAIN) e = labels_simt_t<double, double>(c, seed, gate);
    else if (c->xdt == 2) e = labels_simt_t<float, __nv_bfloat16>(c, seed, gate);
    else e = labels_simt_t<float, float>(c, seed, gate);
    prof_end(c, name);
    c->nlaunch += 1;
    return e;
}

cudaError_t launch_labels_simt(dpmm_ctx* c, uint64_t seed) { return launch_labels_simt_gated(c, seed, nullptr); }

static cudaError_t sort_impl(dpmm_ctx* c, const int* gate) {
    prof_begin(c, "sort");
    hist_kernel<<<c->T_tiles, 256, sizeof(int) * c->K_max, c->stream>>>(c->z, c->N, c->T_tiles, c->K_max, gate,
                                                                         c->hist);
    // tot holds K_max + 1 starts, then the scan's completion counter
    scan_kernel<<<c->K_max, 1024, 0, c->stream>>>(c->hist, c->T_tiles, c->dK, gate, c->tot, c->tot + c->K_max + 1);
    scatter_kernel<<<c->T_tiles, 256, sizeof(int) * 9 * c->K_max, c->stream>>>(c->z, c->N, c->T_tiles, c->hist, c->tot,
                                                                               gate, c->K_max, c->idx);
    prof_end(c, "sort");
    c->nlaunch += 3;
    if (!gate) c->sorted = true;
    return cudaGetLastError();
}

struct SubCfg {
    int P, BT, G;
    size_t smem;
};

template <typename T>
static SubCfg sub_cfg(const dpmm_ctx* c) {
    SubCfg q;
    const StatLayout& L = c->st;
    int P = (int)((64 * 1024) / ((size_t)L.dp * sizeof(T)));
    P = std::max(32, std::min(256, P / 32 * 32));
    int BT = std::max(P, L.nblk);
    BT = std::min(1024, std::max(256, (BT + 31) / 32 * 32));
    q.P = P;
    q.BT = BT;
    // groups of points per register block; every run's end adds the groups up one after
    // another in FP64 (64 cycles each), so no more than 16 (d = 2: one block, 256 groups,
    // took 105 us per statistics step at N = 10,000; 16 groups 19 us)
    q.G = std::max(1, std::min(16, BT / L.nblk));
    size_t head = (size_t)P * L.dp * sizeof(T) + (2 * (size_t)P + 2) * sizeof(int) + P;
    head = (head + 15) / 16 * 16;
    q.smem = head + (size_t)q.G * L.nblk * 32 * sizeof(T);
    return q;
}

static SubCfg sub_cfg_f32(const dpmm_ctx* c, int DV) {
    SubCfg q;
    const StatLayout& L = c->st;
    const size_t stage = ((size_t)2 * DV * DV + 2 * DV + 2 + DV + 4) * 4;
    int P = (int)((64 * 1024) / ((size_t)L.dp * 4));
    P = std::max(32, std::min(256, P / 32 * 32));
    q.P = P;
    q.BT = 256;
    q.G = std::max(1, 256 / L.nblk);
    size_t head = (size_t)P * L.dp * 4 + (2 * (size_t)P + 2) * sizeof(int) + P;
    head = (head + 15) / 16 * 16;
    q.smem = head + stage + 16 + (size_t)q.G * L.nblk * 32 * 4;
    return q;
}

template <typename T, typename XT>
static cudaError_t substats_t(dpmm_ctx* c, uint64_t seed, int draw, const int* gate) {
    SubCfg q = sub_cfg<T>(c);
    SubArgs<T> a;
    a.kind = c->kind;
    a.d = c->d;
    a.xs = c->xs;
    a.N = c->N;
    a.X = c->X;
    a.pv = pview<T>(c);
    a.shift = (const T*)(sizeof(T) == 8 ? (const void*)c->shift_new : (const void*)c->shift32);
    a.z = c->z;
    a.zbar = c->zbar;
    a.idx = c->idx;
    a.dK = c->dK;
    a.diter = c->diter;
    a.gate = gate;
    a.seed = seed;
    a.draw = draw;
    a.P = q.P;
    a.G = q.G;
    a.R = (c->N + c->Gr - 1) / c->Gr;
    a.L = c->st;
    a.rec = c->records;
    if (q.BT <= 256) {
        cudaError_t ea = cudaFuncSetAttribute(substats_kernel<T, XT, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)q.smem);
        if (ea != cudaSuccess) return ea;
        substats_kernel<T, XT, 256><<<c->Gr, q.BT, q.smem, c->stream>>>(a);
    } else {
        cudaError_t ea = cudaFuncSetAttribute(substats_kernel<T, XT, 1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)q.smem);
        if (ea != cudaSuccess) return ea;
        substats_kernel<T, XT, 1024><<<c->Gr, q.BT, q.smem, c->stream>>>(a);
    }
    return cudaGetLastError();
}

static cudaError_t substats_niw64(dpmm_ctx* c, uint64_t seed, int draw, const int* gate) {
    SubCfg q = sub_cfg<double>(c);
    Sub64 b;
    SubArgs<double>& a = b.a;
    a.kind = c->kind;
    a.d = c->d;
    a.xs = c->xs;
    a.N = c->N;
    a.X = c->X;
    a.pv = pview<double>(c);
    a.shift = c->shift_new;
    a.z = c->z;
    a.zbar = c->zbar;
    a.idx = c->idx;
    a.dK = c->dK;
    a.diter = c->diter;
    a.gate = gate;
    a.seed = seed;
    a.draw = draw;
    a.P = std::min(128, q.P);  // find_runs takes a thread per point; two blocks per SM at d = 32
    a.G = q.G;
    a.R = (c->N + c->Gr - 1) / c->Gr;
    a.L = c->st;
    a.rec = c->records;
    b.qW = c->q_W;
    b.qmu = c->q_mu;
    b.qn = c->q_b;
    b.qc = c->q_c;
    const size_t smem = sub64_head(a.P, a.L.dp) + std::max((size_t)q.G * a.L.nblk * 32 * 8, (size_t)c->d * (a.P + 1) * 4);
    auto kern = q.BT <= 256 ? substats_niw64_kernel<256> : substats_niw64_kernel<1024>;
    cudaError_t ea = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (ea != cudaSuccess) return ea;
    kern<<<c->Gr, q.BT, smem, c->stream>>>(b);
    return cudaGetLastError();
}

static cudaError_t combine_impl(dpmm_ctx* c, const int* gate) {
    dim3 grid((c->st.E + 255) / 256, 2 * c->K_max);
    int64_t R = (c->N + c->Gr - 1) / c->Gr;
    combine_kernel<<<grid, 256, 0, c->stream>>>(c->records, c->tot, c->dK, R, c->st.E, c->shift_new, c->shift_stats,
                                                c->d, gate, c->stats);
    return cudaGetLastError();
}

cudaError_t launch_sort(dpmm_ctx* c) { return sort_impl(c, nullptr); }

template <int DV, typename XT>
static cudaError_t substats_f32_t(dpmm_ctx* c, uint64_t seed, int draw, const int* gate) {
    SubCfg q = sub_cfg_f32(c, DV);
    SubArgs<float> a;
    a.kind = c->kind;
    a.d = c->d;
    a.xs = c->xs;
    a.N = c->N;
    a.X = c->X;
    a.pv = pview<float>(c);
    a.shift = c->shift32;
    a.z = c->z;
    a.zbar = c->zbar;
    a.idx = c->idx;
    a.dK = c->dK;
    a.diter = c->diter;
    a.gate = gate;
    a.seed = seed;
    a.draw = draw;
    a.P = q.P;
    a.G = q.G;
    a.R = (c->N + c->Gr - 1) / c->Gr;
    a.L = c->st;
    a.rec = c->records;
    cudaError_t ea = cudaFuncSetAttribute(substats_f32_kernel<DV, XT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)q.smem);
    if (ea != cudaSuccess) return ea;
    substats_f32_kernel<DV, XT><<<c->Gr, q.BT, q.smem, c->stream>>>(a);
    return cudaGetLastError();
}

template <typename XT>
static cudaError_t substats_mult_t(dpmm_ctx* c, uint64_t seed, int draw, const int* gate) {
    const StatLayout& L = c->st;
    // tiles of about 40 KB of rows: four CTAs per SM
    int P = (int)((40 * 1024) / ((size_t)L.dp * 4));
    P = std::max(32, std::min(256, P / 16 * 16));
    const int G = std::max(1, 256 / L.nblk);
    size_t head = (size_t)P * L.dp * 4 + (3 * (size_t)P + 2) * sizeof(int) + P;
    head = (head + 15) / 16 * 16;
    const size_t smem = head + ((size_t)2 * L.dp + 2) * 4 + 16 + (size_t)G * L.nblk * 8 * 4;
    SubArgs<float> a;
    a.kind = c->kind;
    a.d = c->d;
    a.xs = c->xs;
    a.N = c->N;
    a.X = c->X;
    a.pv = pview<float>(c);
    a.shift = c->shift32;
    a.z = c->z;
    a.zbar = c->zbar;
    a.idx = c->idx;
    a.dK = c->dK;
    a.diter = c->diter;
    a.gate = gate;
    a.seed = seed;
    a.draw = draw;
    a.P = P;
    a.G = G;
    a.R = (c->N + c->Gr - 1) / c->Gr;
    a.L = L;
    a.rec = c->records;
    cudaError_t ea = cudaFuncSetAttribute(substats_mult_kernel<XT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (ea != cudaSuccess) return ea;
    substats_mult_kernel<XT><<<c->Gr, 256, smem, c->stream>>>(a);
    return cudaGetLastError();
}

static cudaError_t substats_wide(dpmm_ctx* c, uint64_t seed, int draw, const int* gate) {
    WideArgs w;
    SubArgs<float>& a = w.a;
    a.kind = c->kind;
    a.d = c->d;
    a.xs = c->xs;
    a.N = c->N;
    a.X = c->X;
    a.pv = pview<float>(c);
    a.shift = c->shift32;
    a.z = c->z;
    a.zbar = c->zbar;
    a.idx = c->idx;
    a.dK = c->dK;
    a.diter = c->diter;
    a.gate = gate;
    a.seed = seed;
    a.draw = draw;
    a.P = WP;
    a.G = 1;
    a.R = (c->N + c->Gr - 1) / c->Gr;
    a.L = c->st;
    a.rec = c->records;
    w.starts = c->tot;
    const size_t smem = wide_smem_of(c->st.dp);
    cudaError_t ea = cudaFuncSetAttribute(substats_wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (ea != cudaSuccess) return ea;
    substats_wide_kernel<<<c->Gr, WIDE_T, smem, c->stream>>>(w);
    return cudaGetLastError();
}

// dense multinomial data on the reduced-precision paths: mult_warp_kernel and its compact counts
bool mult_direct(const dpmm_ctx* c) {
    return c->kind == DPMM_PRIOR_DIRICHLET && !c->sparse && c->prec != DPMM_PREC_FP64_PLAIN && c->d <= 256 && c->mcnt &&
           c->xdt == 2 && (c->xs & 7) == 0;
}

static cudaError_t mult_direct_t(dpmm_ctx* c, uint64_t seed, int draw, const int* gate) {
    const dim3 sg((unsigned)std::min(8, (c->d + 1 + 255) / 256), (unsigned)(2 * c->K_max));
    mcnt_zero_kernel<<<sg, 256, 0, c->stream>>>(c->dK, gate, c->d, c->mcnt);
    MwArgs a;
    a.N = c->N;
    a.d = c->d;
    a.xs = c->xs;
    a.X = c->X;
    a.idx = c->idx;
    a.starts = c->tot;
    a.dK = c->dK;
    a.lt = c->q_logtheta;
    a.lc = c->q_c;
    a.diter = c->diter;
    a.seed = seed;
    a.gate = gate;
    a.draw = draw;
    a.zbar = c->zbar;
    a.cnt = c->mcnt;
    const int64_t warps = 24 * (int64_t)c->num_sms;  // three 256-thread blocks per SM
    a.R = std::max<int64_t>(1, (c->N + warps - 1) / warps);
    const unsigned grid = (unsigned)((((c->N + a.R - 1) / a.R) + 7) / 8);
    const int smem = 8 * MW_DEPTH * MW_ROWB;
    cudaError_t e = cudaFuncSetAttribute(mult_warp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    mult_warp_kernel<<<grid, 256, smem, c->stream>>>(a);
    mcnt_fill_kernel<<<sg, 256, 0, c->stream>>>(c->dK, gate, c->st, c->mcnt, c->stats);
    return cudaGetLastError();
}

static cudaError_t substats_dispatch(dpmm_ctx* c, uint64_t seed, int draw, const int* gate) {
    prof_begin(c, draw ? "substats" : "restats");
    cudaError_t e;
    if (mult_direct(c)) {
        e = mult_direct_t(c, seed, draw, gate);
        prof_end(c, draw ? "substats" : "restats");
        c->nlaunch += 3;
        return e;
    }
    const bool mult_fast = c->prec != DPMM_PREC_FP64_PLAIN && c->kind == DPMM_PRIOR_DIRICHLET && c->st.nblk <= 256;
    if (mult_fast) {
        e = c->xdt == 2 ? substats_mult_t<__nv_bfloat16>(c, seed, draw, gate) : substats_mult_t<float>(c, seed, draw, gate);
        prof_end(c, draw ? "substats" : "restats");
        c->nlaunch += 1;
        return e;
    }
    const bool fast = c->prec != DPMM_PREC_FP64_PLAIN && c->kind == DPMM_PRIOR_NIW && c->d <= 64 && c->st.nblk <= 256;
    if (substats_tc_supported(c)) e = launch_substats_tc(c, seed, draw, gate);
    else if (fast && c->d <= 32) e = c->xdt == 2 ? substats_f32_t<32, __nv_bfloat16>(c, seed, draw, gate)
                                             : substats_f32_t<32, float>(c, seed, draw, gate);
    else if (fast) e = c->xdt == 2 ? substats_f32_t<64, __nv_bfloat16>(c, seed, draw, gate)
                                   : substats_f32_t<64, float>(c, seed, draw, gate);
    else if (c->prec != DPMM_PREC_FP64_PLAIN && c->kind == DPMM_PRIOR_NIW && c->d <= 128 && c->st.nblk <= WIDE_T)
        e = substats_wide(c, seed, draw, gate);
    else if (c->prec == DPMM_PREC_FP64_PLAIN && c->kind == DPMM_PRIOR_NIW && c->d > 8) e = substats_niw64(c, seed, draw, gate);
    else if (c->prec == DPMM_PREC_FP64_PLAIN) e = substats_t<double, double>(c, seed, draw, gate);
    else if (c->xdt == 2) e = substats_t<float, __nv_bfloat16>(c, seed, draw, gate);
    else e = substats_t<float, float>(c, seed, draw, gate);
    prof_end(c, draw ? "substats" : "restats");
    c->nlaunch += 1;
    return e;
}

cudaError_t launch_substats(dpmm_ctx* c, uint64_t seed, int draw_zbar) {
    return substats_dispatch(c, seed, draw_zbar, nullptr);
}

cudaError_t launch_combine(dpmm_ctx* c) {
    if (mult_direct(c)) return cudaSuccess;  // the counts went straight to the table
    prof_begin(c, "combine");
    cudaError_t e = combine_impl(c, nullptr);
    prof_end(c, "combine");
    c->nlaunch += 1;
    return e;
}

// statistics recomputed from the labels, only when the split/merge step changed them
cudaError_t launch_restats_gated(dpmm_ctx* c, const int* gate) {
    if (c->sparse) return launch_sparse(c, 0, 2, gate);
    cudaError_t e = sort_impl(c, gate);
    if (e == cudaSuccess) e = substats_dispatch(c, 0, 0, gate);
    if (e == cudaSuccess && !mult_direct(c)) {
        prof_begin(c, "combine");
        e = combine_impl(c, gate);
        prof_end(c, "combine");
        c->nlaunch += 1;
    }
    return e;
}

cudaError_t launch_init_labels(dpmm_ctx* c, uint64_t seed) {
    c->nlaunch += 1;
    init_labels_kernel<<<(unsigned)((c->N + 255) / 256), 256, 0, c->stream>>>(c->N, c->init_K, seed, c->diter, c->z,
                                                                                c->zbar);
    return cudaGetLastError();
}

}  // namespace dpmm
