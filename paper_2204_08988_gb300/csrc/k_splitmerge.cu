// k_splitmerge.cu -- splits and merges (Sec. 4.1, Eqs. sample_splits and
// sample_merges; Sec. 4.3 "a cluster takes part in at most one merge").
//
//   marginal : log f_x(C; lambda) for every cluster and sub-cluster (Dirichlet: and pair),
//              FP64, one CTA per item (NIW: Cholesky log-determinant of Psi_n;
//              Dirichlet-multinomial: lgamma sums).
//   merge    : every proposal's acceptance (many Gaussian merge pairs: upper bounds of the
//              ratio first, the pair's marginal only where they leave it open).
//   decision : walks the proposals in the fixed order (splits by
//              increasing k, then merge pairs in lexicographic order) with the
//              Philox uniforms (tag SPLIT, c0 = k; tag MERGE, c0 = k1, block k2,
//              indices after removing emptied clusters), and writes the relabel map.
//   relabel  : applies it to z, z-bar (sub-labels of split clusters re-drawn, tag
//              RESUB); gated: it returns at once when nothing changed.
#include <math.h>

#include <cmath>
#include <type_traits>

#include "dpmm_internal.cuh"
#include "fp64_chol.cuh"

namespace dpmm {

struct SMArgs {
    const double* stats;
    StatLayout L;
    const double* shift_stats;  // K_max x d
    const double* m0s;          // d (storage coordinates)
    const double* psi0;         // d x d
    const double* beta;         // d
    double kappa0, nu0, logdet_psi0, alpha;
    double log_alpha, lg_alpha, lg_half_alpha;  // log a, lgamma(a), lgamma(a / 2), from the host
    double lmvg_nu0;                            // sum_j lgamma(nu0 / 2 - j / 2), from the host
    double half_d_log_kappa0;                   // d / 2 log kappa0, from the host
    double sum_beta, lg_sum_beta, sum_lg_beta;  // sum beta_j, its lgamma, sum lgamma(beta_j)
    int stage;                                  // statistics blocks staged in shared memory
    int kind, K_max;
    const int* dK;
    float* T32;      // NIW: T_k = Psi0 / 2 + C_k of every cluster in FP32 (K_max x d x d, lower triangle)
    double* xbar;    // K_max x d cluster means
    double* ldT;     // K_max: log det T_k (NaN: not known)
    int exact;       // slots and pairs up to this many: every pair is factorised in FP64 at once
};
// whether marginal_kernel evaluates the pairs itself (else merge_kernel bounds them)
__device__ inline bool pairs_at_once(const SMArgs& a, int K) {
    return a.kind == DPMM_PRIOR_DIRICHLET || 3 * K + K * (K - 1) / 2 <= a.exact;
}

__device__ inline double smv(const SMArgs& a, int k, int h, int j, int l) {
    int e = a.L.ent(j, l);
    if (h >= 0) return a.stats[(size_t)(2 * k + h) * a.L.E + e];
    return a.stats[(size_t)(2 * k) * a.L.E + e] + a.stats[(size_t)(2 * k + 1) * a.L.E + e];
}

// per-slot lgamma table after the log marginals: lg[2 s] = lgamma(n_s),
// lg[2 s + 1] = lgamma(alpha / 2 + n_s)
__host__ __device__ inline size_t lg_offset(int K_max) { return 3 * (size_t)K_max + (size_t)K_max * (K_max - 1) / 2 + 1; }
// then lgamma(n) and lgamma(alpha + n) of every merge pair's n = n_k1 + n_k2 (two per pair)
__host__ __device__ inline size_t lg_pair_offset(int K_max) { return lg_offset(K_max) + 6 * (size_t)K_max; }

__device__ inline void pair_of(int p, int K, int& k1, int& k2) {
    int r = 0, off = 0;
    while (off + (K - r - 1) <= p) {
        off += K - r - 1;
        ++r;
    }
    k1 = r;
    k2 = r + 1 + (p - off);
}

// One item (slot or merge pair) of marginal_kernel, by two warps or more (the last one takes the
// lgamma terms).  Dynamic shared memory: d (d | 1) + 9 d doubles (+ 2 E when the statistics are staged).
// t >= 0: T_t = Psi0 / 2 + C_t of cluster t instead (its entries, the mean and log det T_t).
__device__ __forceinline__ void marginal_item(const SMArgs& a, double* Ltab, int* derr, int K, int e, int t = -1) {
    extern __shared__ double smem[];
    __shared__ double sh[32];
    __shared__ double s_n, s_n1, s_n2;
    const int d = a.L.d, tid = threadIdx.x, nt = blockDim.x;
    int k1, k2, h;
    if (t >= 0) {
        k1 = t;
        k2 = -1;
        h = -1;
    } else if (e < 3 * K) {
        k1 = e / 3;
        k2 = -1;
        h = e % 3 - 1;
    } else {
        pair_of(e - 3 * K, K, k1, k2);
        h = -1;
    }
    double* out = Ltab + (e < 3 * K ? e : 3 * a.K_max + (e - 3 * K));
    // the slot's or the pair's lgamma terms for the Hastings ratios
    double* lgt = Ltab + (e < 3 * K ? lg_offset(a.K_max) + 2 * e : lg_pair_offset(a.K_max) + 2 * (e - 3 * K));
    const double alpha = e < 3 * K ? 0.5 * a.alpha : a.alpha;
    if (a.kind == DPMM_PRIOR_DIRICHLET) {
        if (tid == 32 || tid == 33) {
            const double n = smv(a, k1, h, d, d) + (k2 >= 0 ? smv(a, k2, -1, d, d) : 0.0);
            lgt[tid - 32] = lgamma(tid == 32 ? n : alpha + n);
        }
        // the prior's terms (sum beta, lgamma(sum beta), sum lgamma(beta_j)) come from the host
        double sc = 0.0, acc = 0.0;
        for (int j = tid; j < d; j += nt) {
            double c = smv(a, k1, h, j, d) + (k2 >= 0 ? smv(a, k2, -1, j, d) : 0.0);
            sc += c;
            acc += lgamma(a.beta[j] + c);
        }
        double tot = 0.0;
        // sum counts and lgamma terms over the block (fixed order)
        for (int o = 16; o > 0; o >>= 1) {
            sc += __shfl_xor_sync(0xffffffffu, sc, o);
            acc += __shfl_xor_sync(0xffffffffu, acc, o);
        }
        __shared__ double shc[32], sha[32];
        if ((tid & 31) == 0) {
            shc[tid >> 5] = sc;
            sha[tid >> 5] = acc;
        }
        __syncthreads();
        if (tid == 0) {
            double c = 0.0, l = 0.0;
            for (int w = 0; w < (nt + 31) / 32; ++w) {
                c += shc[w];
                l += sha[w];
            }
            tot = l - a.sum_lg_beta + a.lg_sum_beta - lgamma(a.sum_beta + c);
            *out = tot;
        }
        return;
    }
    const int ld = d | 1;      // odd row stride: column reads without bank conflicts
    double* A = smem;          // d x ld (lower triangle)
    double* piv = A + d * ld;  // pivots of the factorisation
    double* cols = piv + d;    // 8 d: the factorisation's scaled panel columns, and before it
    double* u1 = cols;           // first moments / n of (k1, h), of k2
    double* u2 = u1 + d;
    double* g = u2 + d;          // f (merged mean - m0)
    double* wx = g + d;          // n1 n2 / n (mean 1 - mean 2)
    double* dx = wx + d;         // mean 1 - mean 2
    double* dxb = dx + d;        // merged mean - m0
    double* S1 = cols + 8 * d;   // staged statistics of (k1, h) and of cluster k2 (E each)
    double* S2 = S1 + a.L.E;
    const bool staged = a.stage != 0;
    // Psi0's entries of a thread's first entries, loaded beside the statistics
    constexpr int UB = 5;        // entries a thread at a time
    const int nc = nt - 32, ntri = d * (d + 1) / 2;
    int jj[UB], ll[UB];
    double p0[UB];
    auto psi0_of = [&](int e0) {
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            tri_index(min(e0 + u * nc, ntri - 1), jj[u], ll[u]);  // l <= j: the factorisation reads nothing else
            p0[u] = a.psi0[jj[u] * d + ll[u]];
        }
    };
    if (tid < nc) psi0_of(tid);
    if (staged) {
        stage_slot(a.stats, a.L.E, k1, h, S1);
        if (k2 >= 0) stage_slot(a.stats, a.L.E, k2, -1, S2);
        __syncthreads();
    }
    // M[j][l] (j <= l) of the first and second statistics block
    auto M1 = [&](int j, int l) -> double { return staged ? S1[a.L.ent(j, l)] : smv(a, k1, h, j, l); };
    auto M2 = [&](int j, int l) -> double { return staged ? S2[a.L.ent(j, l)] : smv(a, k2, -1, j, l); };
    __shared__ double s_div[4], s_lg;
    if (tid < 4) {  // 1 / n1, 1 / n2, 1 / n and f, one reciprocal in four lanes
        const double n1 = M1(d, d), n2 = k2 >= 0 ? M2(d, d) : 0.0, n = n1 + n2;
        const double den = tid == 0 ? n1 : tid == 1 ? n2 : tid == 2 ? n : a.kappa0 + n;
        const double num = tid == 3 ? a.kappa0 * n : 1.0;
        s_div[tid] = recip_range(den) ? num * recip_fast(den) : den > 0 ? num * recip_any(den) : 0.0;
        if (tid == 0) {
            s_n1 = n1;
            s_n2 = n2;
            s_n = n;
        }
    }
    __syncthreads();
    const double n1 = s_n1, n2 = s_n2, n = s_n, kn = a.kappa0 + n, nun = a.nu0 + n;
    __shared__ int s_fail;
    if (tid >= nc) {
        // the lgamma terms and log kappa_n, which need n alone, beside the factorisation (a call is a chain of
        // some 6,000 cycles)
        double part = 0.0;
        if (t < 0) {
            if (tid == nt - 1) part = -0.5 * d * log(kn);
            for (int q = tid - nc; q < d + 2; q += 32) {
                const double v = lgamma(q < d ? 0.5 * nun - 0.5 * q : q == d ? n : alpha + n);
                if (q < d) part += v;
                else lgt[q - d] = v;
            }
        }
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        if (tid == nc) s_lg = part;
    } else {
        auto sync = [nc] { asm volatile("bar.sync 1, %0;" ::"r"(nc) : "memory"); };
        const double r1 = s_div[0], r2 = s_div[1], rn = s_div[2], f = s_div[3], w12 = n1 * n2 * rn;
        if (tid == 0) s_fail = 0;
        for (int j = tid; j < d; j += nc) {
            const double v1 = n1 > 0 ? M1(j, d) * r1 : 0.0, v2 = k2 >= 0 && n2 > 0 ? M2(j, d) * r2 : 0.0;
            const double m1 = n1 > 0 ? a.shift_stats[(size_t)k1 * d + j] + v1 : 0.0;
            const double m2 = k2 >= 0 && n2 > 0 ? a.shift_stats[(size_t)k2 * d + j] + v2 : 0.0;
            const double xb = n > 0 ? (n1 * m1 + n2 * m2) * rn : 0.0;
            u1[j] = v1;
            u2[j] = v2;
            dx[j] = m1 - m2;
            wx[j] = w12 * (m1 - m2);
            dxb[j] = xb - a.m0s[j];
            g[j] = f * (xb - a.m0s[j]);
            if (t >= 0) a.xbar[(size_t)t * d + j] = xb;
        }
        sync();
        for (int e0 = tid; e0 < ntri; e0 += UB * nc) {
            if (e0 != tid) psi0_of(e0);
#pragma unroll
            for (int u = 0; u < UB; ++u) {
                if (e0 + u * nc >= ntri) break;
                const int j = jj[u], l = ll[u];
                double v = t >= 0 ? 0.5 * p0[u] : p0[u];
                if (n1 > 0) v += fma(-M1(l, d), u1[j], M1(l, j));
                if (k2 >= 0 && n2 > 0) {
                    v += fma(-M2(l, d), u2[j], M2(l, j));
                    if (n1 > 0) v = fma(wx[j], dx[l], v);
                }
                if (t >= 0) a.T32[(size_t)t * d * d + j * d + l] = (float)v;
                else v = fma(g[j], dxb[l], v);
                A[j * ld + l] = v;
            }
        }
        sync();
        chol_ldl_blk<double>(A, d, ld, piv, cols, cols + 4 * d, nullptr, 0.0, &s_fail, t >= 0 ? nullptr : derr, nc, sync);
        double part = 0.0;
        for (int j = tid; j < d; j += nc) part += log(piv[j]);
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        if ((tid & 31) == 0) sh[tid >> 5] = part;
    }
    __syncthreads();
    if (tid == 0) {
        double s = 0.0;  // log det
        for (int w = 0; w < nc / 32; ++w) s += sh[w];
        if (t >= 0)
            a.ldT[t] = s_fail ? nan("") : s;  // a factorisation that fails says nothing: the pair is factorised itself
        else  // -(nun/2) log|Psi_n| and the multivariate-lgamma ratio; 1.1447298858494002 = log(pi)
            *out = -0.5 * n * d * 1.1447298858494002 - 0.5 * nun * s + s_lg - a.lmvg_nu0 + 0.5 * a.nu0 * a.logdet_psi0 + a.half_d_log_kappa0;
    }
}

// Log marginal likelihoods of every slot (cluster and sub-clusters) and merge pair, or, for
// Gaussian data with many pairs, T_k of every cluster, from which merge_kernel bounds the
// pairs.  An item is a chain of FP64 latencies, so pairs that an SM can take beside the slots
// cost little (d = 32, 60 slots and 190 pairs: 38 us; 50 us before the lookahead factorisation).  The resident blocks
// take the items in turn, so that no block is launched for the slots and pairs beyond K.
constexpr int MARG_T = 160;
__global__ void __launch_bounds__(MARG_T) marginal_kernel(SMArgs a, double* Ltab, int* derr) {
    const int K = *a.dK;
    const bool bound = !pairs_at_once(a, K);
    const int total = 3 * K + (bound ? K : K * (K - 1) / 2);
    for (int e = blockIdx.x; e < total; e += gridDim.x) {
        marginal_item(a, Ltab, derr, K, e, bound && e >= 3 * K ? e - 3 * K : -1);
        __syncthreads();  // shared memory is reused by the next item
    }
}

// The Dirichlet-multinomial log marginals from the sub-cluster counts (Src: the FP32 compact
// table of compressed-row data, or the statistics table of dense data on the reduced-precision
// paths).  Only categories with a nonzero count contribute (for c = 0,
// lgamma(beta_j + c) - lgamma(beta_j) = 0).  The term for count c is read from a table of
// lgamma(beta + c) - lgamma(beta) made on the host when every beta_j is equal and c is below
// its length, and computed otherwise.  Same outputs as marginal_kernel (Ltab), one CTA per
// cluster, sub-cluster and pair.
template <typename Src>
__device__ __forceinline__ void marginal_counts_item(const SMArgs& a, const Src& cnt, const double* lgt, int nlgt,
                                                     const double* lgb, double* Ltab, int K, int e) {
    __shared__ double shc[32], sha[32];
    const int d = a.L.d, tid = threadIdx.x, nt = blockDim.x;
    int k1, k2, h;
    if (e < 3 * K) {
        k1 = e / 3;
        k2 = -1;
        h = e % 3 - 1;
    } else {
        pair_of(e - 3 * K, K, k1, k2);
        h = -1;
    }
    double* out = Ltab + (e < 3 * K ? e : 3 * a.K_max + (e - 3 * K));
    if (tid == 32 || tid == 33) {  // the slot's or the pair's lgamma terms for the Hastings ratios
        if (e < 3 * K) {
            const double ns = smv(a, k1, h, d, d);
            Ltab[lg_offset(a.K_max) + 2 * e + (tid - 32)] = lgamma(tid == 32 ? ns : 0.5 * a.alpha + ns);
        } else {
            const double nm = smv(a, k1, -1, d, d) + smv(a, k2, -1, d, d);
            Ltab[lg_pair_offset(a.K_max) + 2 * (e - 3 * K) + (tid - 32)] = lgamma(tid == 32 ? nm : a.alpha + nm);
        }
    }
    using V = decltype(cnt(0, 0));  // the source's own type: FP32 sums stay off the FP64 pipe
    const int s0 = 2 * k1 + (h < 0 ? 0 : h);
    // compressed rows hold whole counts, which are added as integers (exact, as FP64 adds of them
    // are): a conversion to FP64 and an FP64 add a category kept the two-lane FP64 pipe busy two
    // thirds of the time (d = 20,000, K = 20: 46 us, from 66).  Dense data may hold fractions.
    std::conditional_t<sizeof(V) == 4, unsigned long long, double> si = 0;
    double acc = 0.0;
    for (int j = tid; j < d; j += nt) {
        V c = cnt(s0, j);
        if (h < 0) c += cnt(2 * k1 + 1, j);
        if (k2 >= 0) c += cnt(2 * k2, j) + cnt(2 * k2 + 1, j);  // whole counts: exact
        if (c > V(0)) {
            if constexpr (sizeof(V) == 4) si += (unsigned)c;
            else si += c;
            acc += (lgt && c < (V)nlgt) ? lgt[(int)c] : lgamma(a.beta[j] + (double)c) - lgb[j];
        }
    }
    double sc = (double)si;
    for (int o = 16; o > 0; o >>= 1) {
        sc += __shfl_xor_sync(0xffffffffu, sc, o);
        acc += __shfl_xor_sync(0xffffffffu, acc, o);
    }
    if ((tid & 31) == 0) {
        shc[tid >> 5] = sc;
        sha[tid >> 5] = acc;
    }
    __syncthreads();
    if (tid == 0) {
        double c = 0.0, l = 0.0;
        for (int w = 0; w < (nt + 31) / 32; ++w) {  // fixed order
            c += shc[w];
            l += sha[w];
        }
        *out = l + a.lg_sum_beta - lgamma(a.sum_beta + c);
    }
}

template <typename Src>
__global__ void marginal_counts_kernel(SMArgs a, Src cnt, const double* lgt, int nlgt, const double* lgb, double* Ltab) {
    const int K = *a.dK;
    const int total = 3 * K + K * (K - 1) / 2;
    for (int e = blockIdx.x; e < total; e += gridDim.x) {
        marginal_counts_item<Src>(a, cnt, lgt, nlgt, lgb, Ltab, K, e);
        __syncthreads();  // shared memory is reused by the next item
    }
}

constexpr int DEC_KMAX = 1024;  // K_max <= 1000

struct DecArgs {
    SMArgs s;
    const double* Ltab;
    const uint32_t* diter;
    uint64_t seed;
    int burn_out, labels_ran, sm_enabled, init_mode;
    const int* acc;    // merge_kernel's accept flags
    int* age;          // K_max
    int* dK;
    int* relabel;      // 3 K_max: map_l, map_r, zmode
    int* counters;     // [0] splits [1] merges [2] rejected (K_max) [3] removed [4] changed
    double* shift_new; // K_max x d
    float* shift32;
    int* derr;
};

// Dynamic shared memory: the accept flags (one byte per proposal) when they fit in
// dyn_flags bytes, so that the sequential walk reads shared memory only.  The
// bookkeeping (live clusters, split targets, new ids, ages, relabel maps) is done by
// ballot prefix counts over chunks of 32 clusters in cluster order, which gives the ids
// a sequential walk gives; only the merge walk is sequential (on bit masks for K <= 64).
__global__ void decision_kernel(DecArgs a, int dyn_flags) {
    __shared__ int live[DEC_KMAX], split_to[DEC_KMAX], merged_into[DEC_KMAX], head[DEC_KMAX];
    __shared__ int newid[DEC_KMAX], newid_split[DEC_KMAX], src[DEC_KMAX], nage[DEC_KMAX], cid[DEC_KMAX];
    __shared__ unsigned long long rowm[64];
    __shared__ int s_Kc, s_nsplit, s_nrej, s_nmerge, s_nid;
    extern __shared__ unsigned char flg[];
    const int tid = threadIdx.x, lane = tid & 31;
    const unsigned below = (1u << lane) - 1u;
    const int K = *a.s.dK;
    const int d = a.s.L.d;
    const int nflags = K + K * (K - 1) / 2;
    const bool staged = a.sm_enabled && nflags <= dyn_flags;
    for (int k = tid; k < K; k += blockDim.x) {
        live[k] = a.labels_ran ? (smv(a.s, k, -1, d, d) > 0) : 1;
        nage[k] = a.age[k];
        split_to[k] = -1;
        merged_into[k] = -1;
        head[k] = 0;
    }
    if (staged) {
        for (int q = tid; q < nflags; q += blockDim.x) flg[q] = (unsigned char)(q < K ? a.acc[q] : a.acc[a.s.K_max + q - K]);
    }
    __syncthreads();
    auto acc_split = [&](int k) { return staged ? (int)flg[k] : a.acc[k]; };
    auto acc_merge = [&](int p) { return staged ? (int)flg[K + p] : a.acc[a.s.K_max + p]; };
    // splits: the accepted proposals of live clusters past burn-out, in cluster order, take
    // the ids Kc, Kc + 1, ... below K_max; the ones beyond K_max are rejected
    if (tid < 32) {
        int Kc = 0;
        for (int k0 = 0; k0 < K; k0 += 32) Kc += __popc(__ballot_sync(0xffffffffu, k0 + lane < K && live[k0 + lane]));
        int want = 0, ns = 0;
        if (a.sm_enabled) {
            const int room = a.s.K_max - Kc;
            for (int k0 = 0; k0 < K; k0 += 32) {
                const int k = k0 + lane;
                const bool w = k < K && live[k] && nage[k] >= a.burn_out && acc_split(k);
                const unsigned m = __ballot_sync(0xffffffffu, w);
                const int r = want + __popc(m & below);
                if (w && r < room) split_to[k] = Kc + r;
                want += __popc(m);
            }
            ns = min(want, max(room, 0));
        }
        if (lane == 0) {
            s_Kc = Kc;
            s_nsplit = ns;
            s_nrej = want - ns;
        }
    }
    __syncthreads();
    // merges: for k1 in order, the first eligible k2 > k1 whose proposal is accepted
    // (eligible: live, not split, not merged, not already a merge's head)
    if (tid < 32) {
        int nm = 0;
        if (a.sm_enabled) {
            if (K <= 64) {
                for (int k1 = lane; k1 < K; k1 += 32) {  // bit k2 of row k1: pair (k1, k2) accepted
                    unsigned long long row = 0;
                    const int p0 = k1 * (2 * K - k1 - 1) / 2 - k1 - 1;
                    for (int k2 = k1 + 1; k2 < K; ++k2)
                        if (acc_merge(p0 + k2)) row |= 1ull << k2;
                    rowm[k1] = row;
                }
                unsigned long long el = 0;
                for (int k0 = 0; k0 < K; k0 += 32) {
                    const int k = k0 + lane;
                    el |= (unsigned long long)__ballot_sync(0xffffffffu, k < K && live[k] && split_to[k] < 0) << k0;
                }
                __syncwarp();
                if (lane == 0) {
                    for (int k1 = 0; k1 < K; ++k1) {
                        if (!((el >> k1) & 1ull)) continue;
                        const unsigned long long cand = el & rowm[k1];
                        if (cand) {
                            const int k2 = __ffsll((long long)cand) - 1;
                            merged_into[k2] = k1;
                            head[k1] = 1;
                            el &= ~((1ull << k1) | (1ull << k2));
                            ++nm;
                        }
                    }
                }
            } else {  // 32 candidates at a time by the warp; same outcome as the plain double loop
                auto elig = [&](int k) { return live[k] && split_to[k] < 0 && merged_into[k] < 0 && !head[k]; };
                for (int k1 = 0; k1 < K; ++k1) {
                    if (!elig(k1)) continue;
                    int found = -1;
                    for (int b0 = k1 + 1; b0 < K && found < 0; b0 += 32) {
                        const int k2 = b0 + lane;
                        const bool ok = k2 < K && elig(k2) && acc_merge(k1 * (2 * K - k1 - 1) / 2 + (k2 - k1 - 1));
                        const unsigned m = __ballot_sync(0xffffffffu, ok);
                        if (m) found = b0 + __ffs(m) - 1;
                    }
                    if (found >= 0) {
                        if (lane == 0) {
                            merged_into[found] = k1;
                            head[k1] = 1;
                        }
                        ++nm;
                    }
                    __syncwarp();
                }
            }
        }
        if (lane == 0) s_nmerge = nm;
    }
    __syncthreads();
    // new ids: the clusters that stay (live, not merged away) keep their order, then the
    // second halves of the splits in cluster order; src[new id] = old cluster
    if (tid < 32) {
        int base = 0;
        for (int k0 = 0; k0 < K; k0 += 32) {
            const int k = k0 + lane;
            const bool sv = k < K && live[k] && merged_into[k] < 0;
            const unsigned m = __ballot_sync(0xffffffffu, sv);
            const int q = base + __popc(m & below);
            if (k < K) newid[k] = sv ? q : -1;
            if (sv) src[q] = k;
            base += __popc(m);
        }
        for (int k0 = 0; k0 < K; k0 += 32) {
            const int k = k0 + lane;
            const bool sp = k < K && split_to[k] >= 0;
            const unsigned m = __ballot_sync(0xffffffffu, sp);
            const int q = base + __popc(m & below);
            if (sp) {
                newid_split[k] = q;
                src[q] = k;
            }
            base += __popc(m);
        }
        if (lane == 0) {
            if (base == 0) {  // no cluster holds a point: the statistics disagree with the labels
                atomicExch(a.derr, (int)DPMM_ENUMERIC);
                newid[0] = 0;
                src[0] = 0;
                live[0] = 1;
                base = 1;
            }
            s_nid = base;
        }
    }
    __syncthreads();
    const int nid = s_nid;
    // ages: survivors one sweep older, clusters created by a split or merge start at 0
    for (int q = tid; q < nid; q += blockDim.x) {
        const int k = src[q];
        const bool fresh = split_to[k] >= 0 || head[k];  // both halves of a split, and a merge
        cid[q] = fresh ? 0 : nage[k] + (a.init_mode ? 0 : 1);
    }
    int* map_l = a.relabel;
    int* map_r = a.relabel + a.s.K_max;
    int* zmode = a.relabel + 2 * a.s.K_max;
    for (int k = tid; k < K; k += blockDim.x) {
        if (!live[k]) {
            map_l[k] = map_r[k] = -1;
            zmode[k] = 0;
        } else if (split_to[k] >= 0) {
            map_l[k] = newid[k];
            map_r[k] = newid_split[k];
            zmode[k] = 3;
        } else if (merged_into[k] >= 0) {
            map_l[k] = map_r[k] = newid[merged_into[k]];
            zmode[k] = 2;
        } else if (head[k]) {
            map_l[k] = map_r[k] = newid[k];
            zmode[k] = 1;
        } else {
            map_l[k] = map_r[k] = newid[k];
            zmode[k] = 0;
        }
    }
    if (tid == 0) {
        const int nsplit = s_nsplit, nmerge = s_nmerge;
        a.counters[0] = nsplit;
        a.counters[1] = nmerge;
        a.counters[2] = s_nrej;
        a.counters[3] = K - s_Kc;
        a.counters[4] = (nid != K || nsplit || nmerge) ? 1 : 0;
    }
    __syncthreads();
    const int Kn = nid;
    // the statistics shifts follow their clusters (Gaussian only: the multinomial
    // statistics are not shifted, and d x K can be 20,000 x 100 there)
    if (a.s.kind == DPMM_PRIOR_NIW)
    for (int q = tid; q < Kn * d; q += blockDim.x) {
        int k = q / d, j = q % d;
        double v = a.s.shift_stats[(size_t)src[k] * d + j];
        a.shift_new[(size_t)k * d + j] = v;
        a.shift32[(size_t)k * d + j] = (float)v;
    }
    for (int k = tid; k < Kn; k += blockDim.x) a.age[k] = cid[k];
    __syncthreads();
    if (tid == 0) *a.dK = Kn;
}

// log H of the split of cluster k (Eq. sample_splits) and of the merge of pair p = (k1, k2)
// (Eq. sample_merges) from the tables of marginal_kernel.
__device__ inline double split_ratio(const SMArgs& a, const double* Ltab, int k) {
    const double* lg = Ltab + lg_offset(a.K_max);
    return a.log_alpha + lg[2 * (3 * k + 1)] + Ltab[3 * k + 1] + lg[2 * (3 * k + 2)] + Ltab[3 * k + 2] - lg[2 * (3 * k)] -
           Ltab[3 * k];
}
// what the ratio of a merge takes from its two clusters
__device__ inline double merge_rest(const SMArgs& a, const double* Ltab, int k1, int k2) {
    const double* lg = Ltab + lg_offset(a.K_max);
    return -a.log_alpha - lg[2 * (3 * k1)] - lg[2 * (3 * k2)] - Ltab[3 * k1] - Ltab[3 * k2] + a.lg_alpha +
           lg[2 * (3 * k1) + 1] + lg[2 * (3 * k2) + 1] - 2.0 * a.lg_half_alpha;
}
__device__ inline double merge_ratio(const SMArgs& a, const double* Ltab, int p, int k1, int k2) {
    const double* lgp = Ltab + lg_pair_offset(a.K_max) + 2 * (size_t)p;
    return lgp[0] + Ltab[3 * a.K_max + p] - lgp[1] + merge_rest(a, Ltab, k1, k2);
}

// The FP32 bounds' errors are relative, so a pair that has a diagonal entry of T_1 + T_2 below
// this stays open: denormal numbers lose bits (entries beside such a diagonal lose 2^-149, which
// is 2^-50 of it).
constexpr float MERGE_MIN = 1e-30f;

// A merge is refused whatever its uniform (log u >= -36.8) when an upper bound of log H says so.
// log H falls by nu_n / 2 times whatever log|Psi| grows, so a lower bound ld of the pair's log
// determinant gives one.  In FP64 but for lgammaf and logf; lgm = sum_j lgamma((nu_n - j) / 2).  The
// margin, 60 + 4e-6 of the magnitudes of the terms, covers the FP32 functions (lgammaf: 6 ulp) and
// an ld that is off by 4e-6 (|ld| + d).  False when anything is NaN.
__device__ inline bool refused_at(const SMArgs& a, const double* Ltab, int k1, int k2, double n1, double n2, double ld,
                                  float lgm) {
    const int d = a.L.d;
    const double n = n1 + n2, nun = a.nu0 + n, kn = a.kappa0 + n;
    const double lg = (double)lgammaf((float)n) - (double)lgammaf((float)(a.alpha + n));
    const double L = -0.5 * n * d * 1.1447298858494002 - 0.5 * nun * ld + (double)lgm - (double)(0.5f * d * logf((float)kn)) -
                     a.lmvg_nu0 + 0.5 * a.nu0 * a.logdet_psi0 + a.half_d_log_kappa0;
    const double rest = merge_rest(a, Ltab, k1, k2);
    const double size = 0.6 * n * d + 0.5 * nun * (fabs(ld) + d) + fabs((double)lgm) + 2.0 * fabs((double)lgammaf((float)n)) +
                        fabs(Ltab[3 * k1]) + fabs(Ltab[3 * k2]) + fabs(rest);
    return lg + L + rest + 60.0 + 4e-6 * size < -40.0;
}

__device__ inline float warp_lmvgamma(const SMArgs& a, double n) {  // the sum over j, in every lane
    float v = 0.f;
    for (int j = threadIdx.x & 31; j < a.L.d; j += 32) v += lgammaf((float)(0.5 * (a.nu0 + n) - 0.5 * j));
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// First bound, one warp, no factorisation.  With T_k = Psi0 / 2 + C_k, n = n1 + n2, t = n1 / n,
// delta = xbar1 - xbar2 and w = n1 n2 / n, the pair's scale is Psi = T_1 + T_2 + w delta delta^T + (a
// square), so
//   log|Psi| >= log|T_1 + T_2| + log(1 + w delta^T (T_1 + T_2)^-1 delta),
//   log|T_1 + T_2| >= t log|T_1 / t| + (1 - t) log|T_2 / (1 - t)|   (log det is concave),
//   delta^T M^-1 delta >= (delta^T u)^2 / (u^T M u) for any u        (Cauchy-Schwarz),
// taken at u = delta / diag(M).  The quadratic form is raised by 1e-4 of the sum of its magnitudes
// (at most 800 FP32 terms a lane).  u: d floats of the warp's own.
__device__ inline bool refused_by_means(const SMArgs& a, const double* Ltab, int k1, int k2, double n1, double n2, float* u) {
    const int d = a.L.d, lane = threadIdx.x & 31;
    const float* T1 = a.T32 + (size_t)k1 * d * d;
    const float* T2 = a.T32 + (size_t)k2 * d * d;
    float du = 0.f;
    bool in_range = true;
    for (int j = lane; j < d; j += 32) {
        const float dl = (float)(a.xbar[(size_t)k1 * d + j] - a.xbar[(size_t)k2 * d + j]);
        const float m = T1[j * d + j] + T2[j * d + j], v = dl / m;
        in_range = in_range && m >= MERGE_MIN;
        u[j] = v;
        du = fmaf(dl, v, du);
    }
    __syncwarp();
    if (!__all_sync(0xffffffffu, in_range)) return false;
    float qf = 0.f, qa = 0.f;
#pragma unroll 4
    for (int j = 0; j < d; ++j) {
        const float uj = u[j];
        for (int l = lane; l <= j; l += 32) {
            const float m = (l < j ? 2.f : 1.f) * (T1[j * d + l] + T2[j * d + l]) * uj * u[l];
            qf += m;
            qa += fabsf(m);
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        du += __shfl_xor_sync(0xffffffffu, du, o);
        qf += __shfl_xor_sync(0xffffffffu, qf, o);
        qa += __shfl_xor_sync(0xffffffffu, qa, o);
    }
    __syncwarp();
    const double n = n1 + n2;
    const float t = (float)(n1 / n), den = qf + 1e-4f * qa;
    const float q = 0.999f * du * du / den;  // below delta^T M^-1 delta
    const float ent = -(t * logf(t) + (1.f - t) * log1pf(-t));
    const double ld = n1 / n * a.ldT[k1] + n2 / n * a.ldT[k2] + (double)(d * ent + log1pf((float)(n1 * n2 / n) * q));
    return den > 0.f && q >= 0.f && refused_at(a, Ltab, k1, k2, n1, n2, ld, warp_lmvgamma(a, n));
}

// Second bound, the whole block: log|B| of B = T_1 + T_2 + w delta delta^T by an FP32 LDL
// factorisation of A = B - theta diag(B).  The computed factors are those of A + E with
// |E_jl| <= (d + 24) 2^-24 sqrt(b_jj b_ll) (d + 8 roundings of a sum, 4 ulp a reciprocal, the
// rounding of the entries), so E is at most theta diag(B) for theta = d (d + 24) 2^-24 (1.1 of
// it is taken), what was factorised is at most B, and the pivots' product at most |B|.
// Dynamic shared memory: d (d | 1) + 9 d floats.
__device__ inline bool refused_by_factor(const SMArgs& a, const double* Ltab, int k1, int k2, double n1, double n2, float* sm) {
    const int d = a.L.d, ld = d | 1, tid = threadIdx.x, nt = blockDim.x;
    __shared__ int s_fail, s_ref;
    float* A = sm;
    float* piv = A + d * ld;
    float* cols = piv + d;  // 8 d
    float* dl = cols + 4 * d;
    const float* T1 = a.T32 + (size_t)k1 * d * d;
    const float* T2 = a.T32 + (size_t)k2 * d * d;
    for (int j = tid; j < d; j += nt) dl[j] = (float)(a.xbar[(size_t)k1 * d + j] - a.xbar[(size_t)k2 * d + j]);
    if (tid == 0) s_fail = 0;
    __syncthreads();
    const float w = (float)(n1 * n2 / (n1 + n2)) * 0.9999f;
    const float keep = 1.f - 1.1f * 5.97e-8f * (float)d * (float)(d + 24);
    for (int j = tid >> 5; j < d; j += nt >> 5)
        for (int l = tid & 31; l <= j; l += 32) {
            const float b = T1[j * d + l] + T2[j * d + l] + w * dl[j] * dl[l];
            A[j * ld + l] = l == j ? b * keep : b;
            if (l == j && !(b >= MERGE_MIN)) s_fail = 1;
        }
    __syncthreads();
    chol_ldl_blk<float>(A, d, ld, piv, cols, cols + 4 * d, nullptr, 0.f, &s_fail, nullptr, nt, [] { __syncthreads(); });
    if (tid < 32) {
        // the sum of logarithms and that of their magnitudes m: an ulp a logarithm and 9 additions are
        // below 11 x 2^-24 m, also where the features' units differ so that the logarithms cancel
        float v = 0.f, m = 0.f;
        for (int j = tid; j < d; j += 32) {
            const float t = logf(piv[j]);
            v += t;
            m += fabsf(t);
        }
        for (int o = 16; o > 0; o >>= 1) {
            v += __shfl_xor_sync(0xffffffffu, v, o);
            m += __shfl_xor_sync(0xffffffffu, m, o);
        }
        const bool r = !s_fail && refused_at(a, Ltab, k1, k2, n1, n2, (double)v - 1e-6 * m, warp_lmvgamma(a, n1 + n2));
        if (tid == 0) s_ref = r;
    }
    __syncthreads();
    const bool r = s_ref != 0;
    __syncthreads();  // s_ref and the workspace are written again
    return r;
}

// The two bounds of every pair ahead of merge_kernel: acc[K_max + p] = 0 (refused) or 2 (open).  For
// dimensions whose FP64 factorisation leaves room for one block per SM (d = 128: 142 KB): the
// FP32 one takes half of that, and three of these blocks run side by side.
// Dynamic shared memory: refused_by_factor's.
constexpr int BOUND_W = 4;  // warps

__global__ void __launch_bounds__(32 * BOUND_W) bound_kernel(SMArgs a, const double* Ltab, int labels_ran, int* acc) {
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ int s_open[BOUND_W];
    const int K = *a.dK, d = a.L.d, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (pairs_at_once(a, K)) return;
    const int npairs = K * (K - 1) / 2;
    // a block's warps take pairs far apart: a small cluster's pairs, most likely to be open, are
    // neighbours and go to different blocks
    for (int p0 = blockIdx.x; p0 < npairs; p0 += gridDim.x * BOUND_W) {
        const int p = p0 + warp * gridDim.x;
        bool open = false;
        if (p < npairs) {
            int k1, k2;
            pair_of(p, K, k1, k2);
            const double n1 = smv(a, k1, -1, d, d), n2 = smv(a, k2, -1, d, d);
            open = (n1 > 0 && n2 > 0 && !refused_by_means(a, Ltab, k1, k2, n1, n2, (float*)dyn + warp * d)) ||
                   (!labels_ran && !(n1 > 0 && n2 > 0));
            if (!open && lane == 0) acc[a.K_max + p] = 0;
        }
        if (lane == 0) s_open[warp] = open;
        __syncthreads();
        for (int w = 0; w < BOUND_W; ++w) {
            if (!s_open[w]) continue;  // uniform
            int k1, k2;
            const int q = p0 + w * gridDim.x;
            pair_of(q, K, k1, k2);
            const double n1 = smv(a, k1, -1, d, d), n2 = smv(a, k2, -1, d, d);
            const bool r = refused_by_factor(a, Ltab, k1, k2, n1, n2, (float*)dyn);
            if (threadIdx.x == 0) acc[a.K_max + q] = r ? 0 : 2;
        }
        __syncthreads();  // u and s_open are written again
    }
}

// Every split and merge proposal's acceptance, acc[k] for the split of cluster k and acc[K_max
// + p] for merge pair p (1: accepted if proposed; indices in the Philox counters are those
// after removing emptied clusters).  bounded: bound_kernel has been there.  Many Gaussian pairs (not pairs_at_once): a warp bounds each pair's ratio from the means, the
// block factorises in FP32 what that leaves open, and in FP64 what that leaves open; the FP64
// factorisation of every pair was the step's cost (d = 128, K = 64: 2,016 pairs and 192 slots
// 6.0 ms; now 0.6 ms for the slots and 0.8 ms for the pairs).
// Dynamic shared memory: marginal_item's; the bounds' u (a row of d floats per warp) share it.
constexpr int MERGE_W = 8;  // warps

__global__ void __launch_bounds__(32 * MERGE_W) merge_kernel(SMArgs a, double* Ltab, const uint32_t* diter, uint64_t seed,
                                                              int labels_ran, int* acc, int* derr, int bounded) {
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ short s_cid[DEC_KMAX];  // index after removing the empty clusters; -1: empty
    __shared__ int s_open[MERGE_W];
    const int K = *a.dK, d = a.L.d, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nt = 32 * MERGE_W, npairs = K * (K - 1) / 2;
    const bool once = pairs_at_once(a, K);
    // blocks with work (acceptances alone: a proposal per thread); the others leave at once
    const int nb = once ? min((int)gridDim.x, (max(K, npairs) + nt - 1) / nt) : (int)gridDim.x;
    if ((int)blockIdx.x >= nb) return;
    if (warp == 0)
        for (int q0 = 0, base = 0; q0 < K; q0 += 32) {
            const int q = q0 + lane;
            const bool lv = q < K && (!labels_ran || smv(a, q, -1, d, d) > 0);
            const unsigned m = __ballot_sync(0xffffffffu, lv);
            if (q < K) s_cid[q] = lv ? (short)(base + __popc(m & ((1u << lane) - 1u))) : (short)-1;
            base += __popc(m);
        }
    __syncthreads();
    const Key key{seed, diter[0], diter[1], diter[2]};
    // log u < lH; no logarithm where it cannot change the outcome (-36.8 <= log u < 0)
    auto accept = [&](double lH, uint32_t c0, uint32_t tag, uint32_t blk) -> int {
        if (lH >= 0.0) return 1;
        if (!(lH > -40.0)) return 0;
        return log(d_uniform(key, c0, tag, blk)) < lH;
    };
    for (int k = blockIdx.x * nt + tid; k < K; k += nb * nt)
        acc[k] = s_cid[k] >= 0 && smv(a, k, 0, d, d) >= 1 && smv(a, k, 1, d, d) >= 1
                     ? accept(split_ratio(a, Ltab, k), (uint32_t)s_cid[k], TAG_SPLIT, 0) : 0;
    if (once) {
        for (int p = blockIdx.x * nt + tid; p < npairs; p += nb * nt) {
            int k1, k2;
            pair_of(p, K, k1, k2);
            acc[a.K_max + p] = s_cid[k1] >= 0 && s_cid[k2] >= 0
                                   ? accept(merge_ratio(a, Ltab, p, k1, k2), (uint32_t)s_cid[k1], TAG_MERGE, (uint32_t)s_cid[k2]) : 0;
        }
    } else {
        for (int p0 = blockIdx.x; p0 < npairs; p0 += gridDim.x * MERGE_W) {
            const int p = p0 + warp * gridDim.x;
            bool open = false;
            if (p < npairs) {
                int k1, k2;
                pair_of(p, K, k1, k2);
                if (bounded)
                    open = acc[a.K_max + p] == 2;
                else if (s_cid[k1] >= 0 && s_cid[k2] >= 0)
                    open = !refused_by_means(a, Ltab, k1, k2, smv(a, k1, -1, d, d), smv(a, k2, -1, d, d), (float*)dyn + warp * d);
                if (!open && lane == 0) acc[a.K_max + p] = 0;
            }
            if (lane == 0) s_open[warp] = open;
            __syncthreads();
            for (int w = 0; w < MERGE_W; ++w) {
                if (!s_open[w]) continue;  // uniform
                const int q = p0 + w * gridDim.x;
                int k1, k2, ok = 0;
                pair_of(q, K, k1, k2);
                if (bounded ||
                    !refused_by_factor(a, Ltab, k1, k2, smv(a, k1, -1, d, d), smv(a, k2, -1, d, d), (float*)dyn)) {
                    marginal_item(a, Ltab, derr, K, 3 * K + q);
                    __syncthreads();
                    ok = accept(merge_ratio(a, Ltab, q, k1, k2), (uint32_t)s_cid[k1], TAG_MERGE, (uint32_t)s_cid[k2]);
                }
                if (tid == 0) acc[a.K_max + q] = ok;
            }
            __syncthreads();  // u and s_open are written again
        }
    }
}

__global__ void relabel_kernel(int64_t N, const int* relabel, int Kmax, const int* gate, const uint32_t* diter,
                               uint64_t seed, int32_t* z, uint8_t* zbar, int* derr) {
    if (*gate == 0) return;
    const Key key{seed, diter[0], diter[1], diter[2]};
    // grid-stride: the launch is one wave, so that the usual gated-off launch is cheap
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        int k = z[i];
        const int h = zbar[i];
        if ((unsigned)k >= (unsigned)Kmax) {  // never for consistent state: keep memory safe, report
            atomicExch(derr, (int)DPMM_ENUMERIC);
            k = 0;
        }
        const int mode = relabel[2 * Kmax + k];
        int nz = h ? relabel[Kmax + k] : relabel[k];
        if (nz < 0) {  // a point in a cluster counted as empty
            atomicExch(derr, (int)DPMM_ENUMERIC);
            nz = 0;
        }
        z[i] = nz;
        if (mode == 1) zbar[i] = 0;
        else if (mode == 2) zbar[i] = 1;
        else if (mode == 3) zbar[i] = d_uniform(key, (uint32_t)i, TAG_RESUB, 0) < 0.5 ? 0 : 1;
    }
}

__global__ void advance_kernel(uint32_t* diter) { *diter += 1; }

static SMArgs sm_args(dpmm_ctx* c) {
    SMArgs a;
    a.stats = c->stats;
    a.L = c->st;
    a.shift_stats = c->shift_stats;
    a.m0s = c->center + c->d;
    a.psi0 = c->center + 2 * c->d;
    a.beta = c->center + c->d;
    a.kappa0 = c->kappa0;
    a.nu0 = c->nu0;
    a.logdet_psi0 = c->logdet_psi0;
    a.alpha = c->alpha;
    a.log_alpha = std::log(c->alpha);
    a.lg_alpha = std::lgamma(c->alpha);
    a.lg_half_alpha = std::lgamma(0.5 * c->alpha);
    a.lmvg_nu0 = 0.0;
    for (int j = 0; j < c->d; ++j) a.lmvg_nu0 += std::lgamma(0.5 * c->nu0 - 0.5 * j);
    a.half_d_log_kappa0 = 0.5 * c->d * std::log(c->kappa0);
    a.sum_beta = a.lg_sum_beta = a.sum_lg_beta = 0.0;
    if (c->kind == DPMM_PRIOR_DIRICHLET) {
        for (double b : c->beta) {
            a.sum_beta += b;
            a.sum_lg_beta += std::lgamma(b);
        }
        a.lg_sum_beta = std::lgamma(a.sum_beta);
    }
    // in the ranges' records, which have been added up: 8 (d + 1) + 4 d^2 of their 16 E bytes a cluster
    a.xbar = c->records;
    a.ldT = a.xbar + (size_t)c->K_max * c->d;
    a.T32 = (float*)(a.ldT + c->K_max);
    a.stage = 0;
    a.exact = 0;
    a.kind = c->kind;
    a.K_max = c->K_max;
    a.dK = c->dK;
    return a;
}

cudaError_t launch_restats_gated(dpmm_ctx* c, const int* gate);

// the marginals and every proposal's acceptance
static cudaError_t launch_proposals(dpmm_ctx* c, SMArgs& s, uint64_t seed, int labels_ran) {
    // the Dirichlet marginal needs no matrix workspace; the NIW one stages the two statistics
    // blocks it reads when they fit
    size_t smi = 0;
    if (c->kind == DPMM_PRIOR_NIW) {
        smi = sizeof(double) * ((size_t)c->d * (c->d | 1) + 9 * c->d);
        const size_t st = smi + sizeof(double) * 2 * (size_t)c->st.E;
        if (st <= 160 * 1024) {
            smi = st;
            s.stage = 1;
        }
    }
    if (smi > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(marginal_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smi);
        if (e != cudaSuccess) return e;
    }
    // one wave of resident blocks, each taking items in turn (the items beyond the current K
    // launch no block)
    auto waves = [&](const void* fn, int threads, size_t smem, int items) {
        int per = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, threads, smem) != cudaSuccess || per < 1) {
            cudaGetLastError();
            per = 1;
        }
        return (unsigned)std::max<int64_t>(1, std::min<int64_t>(items, (int64_t)per * c->num_sms));
    };
    const int pairs = c->K_max * (c->K_max - 1) / 2, all = 3 * c->K_max + pairs;
    // two items an SM where two fit it side by side (their chains of latencies overlap)
    s.exact = c->num_sms * (smi <= 100 * 1024 ? 2 : 1);
    const bool bounds = c->kind == DPMM_PRIOR_NIW && all > s.exact;  // else every pair is evaluated with the slots
    prof_begin(c, "marginal");
    if (c->sparse)
        marginal_counts_kernel<CountsF32>
            <<<waves((const void*)marginal_counts_kernel<CountsF32>, 256, 0, all), 256, 0, c->stream>>>(
                s, CountsF32{c->sp_cc, c->d}, c->sp_lgt, c->sp_lgt ? SP_LGT : 0, c->sp_lgb, c->Ltab);
    else if (c->kind == DPMM_PRIOR_DIRICHLET && c->prec != DPMM_PREC_FP64_PLAIN)  // dense counts
        marginal_counts_kernel<CountsStats>
            <<<waves((const void*)marginal_counts_kernel<CountsStats>, 256, 0, all), 256, 0, c->stream>>>(
                s, CountsStats{c->stats, c->st}, c->sp_lgt, c->sp_lgt ? SP_LGT : 0, c->sp_lgb, c->Ltab);
    else
        marginal_kernel<<<waves((const void*)marginal_kernel, MARG_T, smi, bounds ? std::max(4 * c->K_max, s.exact) : all),
                          MARG_T, smi, c->stream>>>(s, c->Ltab, c->derr);
    prof_end(c, "marginal");
    c->nlaunch += 1;
    prof_begin(c, "hastings");
    cudaError_t ea = cudaFuncSetAttribute(merge_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smi);
    if (ea != cudaSuccess) return ea;
    const int bounded = bounds && smi > 100 * 1024;
    if (bounded) {
        const size_t bs = sizeof(float) * ((size_t)c->d * (c->d | 1) + 9 * c->d);
        cudaError_t e = cudaFuncSetAttribute(bound_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bs);
        if (e != cudaSuccess) return e;
        bound_kernel<<<waves((const void*)bound_kernel, 32 * BOUND_W, bs, (pairs + BOUND_W - 1) / BOUND_W), 32 * BOUND_W, bs,
                       c->stream>>>(s, c->Ltab, labels_ran, c->acc);
        c->nlaunch += 1;
    }
    const int items = std::max(1, bounds ? (pairs + MERGE_W - 1) / MERGE_W : (pairs + 32 * MERGE_W - 1) / (32 * MERGE_W));
    merge_kernel<<<waves((const void*)merge_kernel, 32 * MERGE_W, smi, items), 32 * MERGE_W, smi, c->stream>>>(
        s, c->Ltab, c->diter, seed, labels_ran, c->acc, c->derr, bounded);
    prof_end(c, "hastings");
    c->nlaunch += 1;
    return cudaGetLastError();
}

cudaError_t launch_splitmerge(dpmm_ctx* c, uint64_t seed, int labels_ran, int sm_enabled) {
    SMArgs s = sm_args(c);
    DecArgs a;
    a.acc = c->acc;
    a.Ltab = c->Ltab;
    a.diter = c->diter;
    a.seed = seed;
    a.burn_out = c->burn_out;
    a.sm_enabled = sm_enabled;
    a.init_mode = (labels_ran == 2);
    a.labels_ran = labels_ran ? 1 : 0;
    a.age = c->age;
    a.dK = c->dK;
    a.relabel = c->relabel;
    a.counters = c->counters;
    a.shift_new = c->shift_new;
    a.shift32 = c->shift32;
    a.derr = c->derr;
    if (sm_enabled) {
        const cudaError_t e = launch_proposals(c, s, seed, a.labels_ran);
        if (e != cudaSuccess) return e;
    }
    a.s = s;
    prof_begin(c, "decision");
    const int dyn = 32 * 1024;
    cudaError_t ea = cudaFuncSetAttribute(decision_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);
    if (ea != cudaSuccess) return ea;
    decision_kernel<<<1, 256, dyn, c->stream>>>(a, dyn);
    prof_end(c, "decision");
    c->nlaunch += 1;
    return cudaGetLastError();
}

cudaError_t launch_relabel(dpmm_ctx* c, uint64_t seed) {
    prof_begin(c, "relabel");
    const unsigned grid = (unsigned)std::min<int64_t>((c->N + 255) / 256, 8 * (int64_t)c->num_sms);
    relabel_kernel<<<grid, 256, 0, c->stream>>>(c->N, c->relabel, c->K_max, c->counters + 4,
                                                                         c->diter, seed, c->z, c->zbar, c->derr);
    prof_end(c, "relabel");
    c->nlaunch += 1;
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = launch_restats_gated(c, c->counters + 4);
    return e;
}

cudaError_t launch_advance(dpmm_ctx* c) {
    advance_kernel<<<1, 1, 0, c->stream>>>(c->diter);
    c->nlaunch += 1;
    return cudaGetLastError();
}

}  // namespace dpmm
