// k_noalloc.cu -- sufficient statistics of given labels without any allocation.
//
// Some callers cannot allocate device memory at the point where they need the
// statistics: an application that reserves the GPU's memory up front in its own pool
// and forbids any later cudaMalloc (a serving process that owns all of HBM, a host
// framework whose plug-ins must not allocate), or latency-critical code that must not
// take the implicit device-wide synchronisation a cudaMalloc/cudaFree can cause.  This
// entry point computes, for every sub-cluster (k, h), the count, the sum of x and the
// sum of x x^T of the points labelled (z = k, zbar = h), using only the caller's
// buffers and a fixed scratch array that lives in this library's device image.  The
// scratch (32 x 2 NA_KMAX x NA_EMAX doubles = 5.6 MiB) is held by every GPU that
// loads the library until the process exits.
#include <cuda.h>

#include <algorithm>
#include <mutex>

#include "dpmm_internal.cuh"

namespace dpmm {

constexpr int NA_RANGES = 32;  // the points are cut into this many ranges, each into tiles
constexpr int NA_KMAX = 16;    // clusters
constexpr int NA_DMAX = 32;    // dimension
constexpr int NA_P = 128;      // points per tile
constexpr int NA_EMAX = 16 * (((NA_DMAX + 4) / 4) * ((NA_DMAX + 4) / 4 + 1) / 2);  // 720 entries
constexpr int NA_W = 8;        // warps per block
constexpr int NA_Q = 4;        // tiles whose labels a warp scans at a time
constexpr int NA_D = 6;        // rows in flight per warp (8 spill registers at d > 16)
constexpr int NA_CARRY = 640;  // additions to a sum before its words are made apart again
constexpr int NA_ROW = 52;     // floats of a staged row: x, then its first d / 2 + 1 values again
constexpr size_t NA_SCRATCH = (size_t)32 * 2 * NA_KMAX * NA_EMAX;  // doubles

static __device__ __align__(256) double g_na_scratch[NA_SCRATCH];

// Two FP32 values in one register pair: the packed instructions do two lanes' work each.
typedef unsigned long long f2;
__device__ __forceinline__ f2 f2_pack(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 f2_unpack(f2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Knuth's two-sum: a becomes a + b rounded; its error, which is returned, is exact
__device__ __forceinline__ f2 f2_two_sum(f2& a, f2 b) {
    const f2 t = f2_add(a, b), bb = f2_sub(t, a);
    const f2 err = f2_add(f2_sub(a, f2_sub(t, bb)), f2_sub(b, bb));
    a = t;
    return err;
}

// Two sums, each of three FP32 words: the errors of s are added up exactly in c, those of c in e.
// With NA_CARRY = 640 additions from one carry to the next, |c| <= 641 x 2^-24 S and |e| <= 640 x 641 x
// 2^-48 S (S: the largest partial sum), so an addition to e loses less than 2^-53 S, which is what
// one to an FP64 sum may lose.
struct NaSum {
    f2 s, c, e;
    __device__ void zero() { s = c = e = 0ull; }
    __device__ void add(f2 a) { e = f2_add(e, f2_two_sum(c, f2_two_sum(s, a))); }
    __device__ void carry() {  // the same sum with |c| <= 2^-24 |s|, |e| <= 2^-24 |c|
        const f2 t = f2_two_sum(c, e);
        c = f2_two_sum(s, c);
        e = f2_two_sum(c, t);
    }
    __device__ double2 value() const {
        const float2 x = f2_unpack(s), y = f2_unpack(c), z = f2_unpack(e);
        return make_double2((double)x.x + ((double)y.x + (double)z.x), (double)x.y + ((double)y.y + (double)z.y));
    }
    __device__ bool bad() const {
        const float2 x = f2_unpack(s), y = f2_unpack(c), z = f2_unpack(e);
        return !isfinite(x.x) || !isfinite(y.x) || !isfinite(z.x) || !isfinite(x.y) || !isfinite(y.y) || !isfinite(z.y);
    }
};
struct NaDouble {
    double2 v;
    __device__ void zero() { v = make_double2(0.0, 0.0); }
    __device__ void carry() {}
    __device__ void add(f2 a) {
        const float2 x = f2_unpack(a);
        v.x += (double)x.x;
        v.y += (double)x.y;
    }
    __device__ double2 value() const { return v; }
    __device__ bool bad() const { return false; }
};

struct NaArgs {
    const float* X;
    int64_t N;
    int d;
    const int32_t* z;
    const uint8_t* zbar;
    int K, G;    // slices
    int W;       // FP32 groups of a tile's points of one slot
    double* scratch;
};

// The sums of one slot: sum x_j x_(j + t mod d) for t = 0 .. d / 2 (every unordered pair of
// features once, lane j), sum x_j, and the count.  ES doubles per (slice, slot).
__host__ __device__ inline int na_entries(int d) { return (d / 2 + 2) * d + 1; }

// Pass 1: block (s, g) sums the points of slot s = 2k + h among the tiles of slice g, each
// warp in tiles of its own.  A warp scans four tiles' labels by ballots (every slot's block
// reads them: 5 bytes a point from L2) and then takes its slot's own rows one after another,
// so X crosses DRAM once: lane j holds x_j, and its partners x_(j + t) come from the row
// staged in shared memory, NA_D rows being loaded while as many are added up.
// What bounds it is the precision: a tile's points of one slot are summed in FP32 (point q
// in group q mod W), and the groups' sums are added with the precision of FP64.  On the FP64 pipe
// that is one conversion and one add per entry and group at two lanes an SM (2.3 ms at d = 32,
// N = 1e6); as three FP32 words it is 13 FP32 adds.  A sum that overflows or meets an infinity or
// NaN makes the block start over in FP64.
// Measured at d = 32, K = 16, N = 1e6: 0.37 ms (0.51 with 8 rows in flight, which spill; 0.27 with two words,
// 48 bits, whose second loses bits with the number of additions); 0.46 ms with two words as 4 x 4
// register blocks over staged tiles (290 million instructions, half of them loops over tiles of four
// points); 25.4 ms for 32 blocks that took a tile's 32 slots in turn, two block barriers each.
template <int T, typename Acc>  // T: odd, at least d / 2 + 1
__device__ __forceinline__ bool na_block(const NaArgs& a, float* row, int* list, double* red) {
    constexpr int NP = (T + 1) / 2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int d = a.d, S = 2 * a.K, s = blockIdx.x, g = blockIdx.y, W = a.W;
    Acc acc[NP];  // t = 2 p and 2 p + 1; the last one's second: sum x_j
    f2 f[NP];     // the group in hand
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        acc[p].zero();
        f[p] = 0ull;
    }
    unsigned long long count = 0;
    int since = 0;  // additions since the last carry
    const int wm = 65536 / W + 1;  // n * wm >> 16 = n / W for 0 <= n <= 128, W <= 256
    const int64_t R = (a.N + NA_RANGES - 1) / NA_RANGES;
    const unsigned Tr = (unsigned)((R + NA_P - 1) / NA_P), tiles = NA_RANGES * Tr;  // tiles per range, in all
    const unsigned per = (tiles + a.G - 1) / a.G, ta = g * per, tb = min(tiles, ta + per);
    const int64_t base = (int64_t)(ta / Tr) * R + (ta % Tr) * NA_P;  // the slice's first point
    const float* Xb = a.X + base * d + (lane < d ? lane : 0);
    float* mine = row + lane;
    const bool again = lane < d && lane <= d / 2;  // x_j is x_(j + d) of the wrapped row
    for (unsigned t0 = ta + NA_Q * warp; t0 < tb; t0 += NA_Q * NA_W) {
        int zi[NA_Q][NA_P / 32], hi[NA_Q][NA_P / 32], off[NA_Q];
#pragma unroll
        for (int u = 0; u < NA_Q; ++u) {
            const unsigned t = t0 + u, r = t / Tr;
            const int64_t i0 = (int64_t)r * R + (int64_t)(t % Tr) * NA_P;
            const int64_t i1 = t < tb ? min(min(a.N, (int64_t)(r + 1) * R), i0 + NA_P) : 0;
            off[u] = (int)(i0 - base);
#pragma unroll
            for (int q = 0; q < NA_P / 32; ++q) {
                const int64_t i = i0 + 32 * q + lane;
                zi[u][q] = i < i1 ? __ldg(a.z + i) : -1;
                hi[u][q] = i < i1 ? (int)__ldg(a.zbar + i) : 2;
            }
        }
        // the slot's points of the four tiles, group by group; the sign bit marks a group's first
        int n = 0;
        __syncwarp();
#pragma unroll
        for (int u = 0; u < NA_Q; ++u) {
            unsigned m[NA_P / 32];
            int nu = 0;
#pragma unroll
            for (int q = 0; q < NA_P / 32; ++q) {  // labels outside [0, K) x {0, 1} match no slot
                m[q] = __ballot_sync(0xffffffffu, zi[u][q] == (s >> 1) && hi[u][q] == (s & 1));
                nu += __popc(m[q]);
            }
            const int nq = nu * wm >> 16, nr = nu - nq * W;
            int r0 = 0;
#pragma unroll
            for (int q = 0; q < NA_P / 32; ++q) {
                if ((m[q] >> lane) & 1u) {
                    const int r = r0 + __popc(m[q] & ((1u << lane) - 1u));
                    const int k = r * wm >> 16, gr = r - k * W;  // r / W and r mod W
                    list[n + gr * nq + min(gr, nr) + k] = (off[u] + 32 * q + lane) | (k == 0 ? 0x80000000 : 0);
                }
                r0 += __popc(m[q]);
            }
            n += nu;
        }
        count += n;
        if (since + n >= NA_CARRY) {  // n <= 512; the last group is added after the loop
#pragma unroll
            for (int p = 0; p < NP; ++p) acc[p].carry();
            since = 0;
        }
        since += n;
        __syncwarp();
        float x[NA_D];
        auto fetch = [&](int q0) {
#pragma unroll
            for (int q = 0; q < NA_D; ++q)
                x[q] = q0 + q < n ? __ldg(Xb + (int64_t)(list[q0 + q] & 0x7fffffff) * d) : 0.f;
        };
        fetch(0);
        for (int q0 = 0; q0 < n; q0 += NA_D) {
            __syncwarp();
#pragma unroll
            for (int q = 0; q < NA_D; ++q) {
                if (lane < d) mine[q * NA_ROW] = x[q];
                if (again) mine[q * NA_ROW + d] = x[q];
            }
            __syncwarp();
            if (q0 + NA_D < n) fetch(q0 + NA_D);
            for (int q = 0; q < min(NA_D, n - q0); ++q) {
                const float* v = mine + q * NA_ROW;
                f2 pr[NP];
#pragma unroll
                for (int p = 0; p < NP; ++p) pr[p] = f2_pack(v[2 * p], p + 1 < NP ? v[2 * p + 1] : 1.f);
                const f2 xj = f2_pack(v[0], v[0]);
                if (list[q0 + q] < 0) {  // a new group: the last one's sums are complete
#pragma unroll
                    for (int p = 0; p < NP; ++p) {
                        acc[p].add(f[p]);
                        f[p] = f2_mul(xj, pr[p]);
                    }
                } else {
#pragma unroll
                    for (int p = 0; p < NP; ++p) f[p] = f2_fma(xj, pr[p], f[p]);
                }
            }
        }
    }
#pragma unroll
    for (int p = 0; p < NP; ++p) acc[p].add(f[p]);
    bool bad = false;
#pragma unroll
    for (int p = 0; p < NP; ++p) bad = bad || acc[p].bad();
    if (__syncthreads_or(lane < d && bad)) return false;
    // the warps' sums in warp order: red[warp][t][j], then the counts
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        const double2 v = acc[p].value();
        red[(warp * (T + 1) + 2 * p) * 32 + lane] = v.x;
        red[(warp * (T + 1) + 2 * p + 1) * 32 + lane] = v.y;
    }
    double* cnt = red + NA_W * (T + 1) * 32;
    if (lane == 0) cnt[warp] = (double)count;
    __syncthreads();
    const int ES = na_entries(d), ns = d / 2 + 1;
    double* out = a.scratch + ((size_t)g * S + s) * ES;
    for (int e = threadIdx.x; e < ES; e += 32 * NA_W) {
        const int t = e / d, j = e % d;
        double v = 0.0;
        for (int w = 0; w < NA_W; ++w)
            v += e == ES - 1 ? cnt[w] : red[(w * (T + 1) + (t < ns ? t : T)) * 32 + j];
        out[e] = v;
    }
    return true;
}

template <int T>
__global__ void __launch_bounds__(32 * NA_W, 2) na_partial_kernel(NaArgs a) {
    constexpr int LIST = NA_Q * NA_P, RED = NA_W * (T + 1) * 32 + NA_W;
    constexpr size_t BYTES = (size_t)NA_W * (LIST * 4 + NA_D * NA_ROW * 4);
    __shared__ __align__(16) unsigned char sm[BYTES > RED * 8 ? BYTES : RED * 8];
    int* list = (int*)sm + (threadIdx.x >> 5) * LIST;
    float* row = (float*)((int*)sm + NA_W * LIST) + (threadIdx.x >> 5) * (NA_D * NA_ROW);
    for (int e = threadIdx.x & 31; e < NA_D * NA_ROW; e += 32) row[e] = 0.f;  // what no feature fills
    __syncwarp();
    if (na_block<T, NaSum>(a, row, list, (double*)sm)) return;
    for (int e = threadIdx.x & 31; e < NA_D * NA_ROW; e += 32) row[e] = 0.f;
    __syncthreads();
    na_block<T, NaDouble>(a, row, list, (double*)sm);
}

// Pass 2: the slices' sums of 32 entries of slot s, eight partial sums each (slice g in
// partial sum g mod 8, added in order: deterministic), unpacked to n, sum x, sum x x^T.
__global__ void __launch_bounds__(256) na_combine_kernel(int d, int G, int K, const double* scratch, double* n_out,
                                                         double* sx_out, double* sxx_out) {
    __shared__ double part[8][32];
    const int s = blockIdx.x, S = 2 * K, ES = na_entries(d);
    const int e = blockIdx.y * 32 + (threadIdx.x & 31), p = threadIdx.x >> 5;
    double v = 0.0;
    if (e < ES)
        for (int g = p; g < G; g += 8) v += scratch[((size_t)g * S + s) * ES + e];
    part[p][threadIdx.x & 31] = v;
    __syncthreads();
    if (p != 0 || e >= ES) return;
    v = 0.0;
    for (int q = 0; q < 8; ++q) v += part[q][threadIdx.x];
    const int t = e / d, j = e % d;
    if (e == ES - 1) {
        n_out[s] = v;
    } else if (t > d / 2) {
        sx_out[(size_t)s * d + j] = v;
    } else if (2 * t < d || j < t) {  // t = d / 2 meets every pair twice
        const int l = (j + t) % d;
        sxx_out[((size_t)s * d + j) * d + l] = v;
        sxx_out[((size_t)s * d + l) * d + j] = v;
    }
}

// The scratch address is looked up (cudaGetSymbolAddress) once per device and per
// context: the array sits at a different address in every context the module is loaded
// into, so the cache is keyed by the context current at the call (cuCtxGetCurrent,
// resolved through the runtime's driver entry point), not by the device ordinal alone.
typedef CUresult (*CtxGetCurrentFn)(CUcontext*);
static std::mutex g_na_mu;
static struct {
    CUcontext ctx;
    void* ptr;
} g_na_cache[128];

static CUcontext na_current_context() {
    static CtxGetCurrentFn fn = nullptr;
    static bool looked = false;
    if (!looked) {
        looked = true;
        cudaDriverEntryPointQueryResult q;
        void* p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (CtxGetCurrentFn)p;
    }
    CUcontext cx = nullptr;
    if (fn && fn(&cx) != CUDA_SUCCESS) cx = nullptr;
    return cx;
}

}  // namespace dpmm

using namespace dpmm;

extern "C" dpmm_status dpmm_suffstats_noalloc(const float* X, int64_t N, int d, const int32_t* z,
                                              const uint8_t* zbar, int K, double* n_out, double* sx_out,
                                              double* sxx_out, void* stream) {
    if (!X || !z || !zbar || !n_out || !sx_out || !sxx_out) return DPMM_EINVAL;
    if (N < 1 || d < 1 || d > NA_DMAX || K < 1 || K > NA_KMAX) return DPMM_EINVAL;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 128) return DPMM_ECUDA;
    double* scratch = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_na_mu);
        const CUcontext cx = na_current_context();
        if (!g_na_cache[dev].ptr || !cx || g_na_cache[dev].ctx != cx) {  // set-up, with that device current
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, g_na_scratch) != cudaSuccess || !p) return DPMM_ECUDA;
            // the lookup has made the runtime's context current if none was
            g_na_cache[dev].ctx = na_current_context();
            g_na_cache[dev].ptr = p;
        }
        scratch = (double*)g_na_cache[dev].ptr;
    }
    cudaStream_t s = (cudaStream_t)stream;
    // slices: about eight blocks per SM over the 2K slots (two are resident at a time, and a
    // large cluster's blocks take longer than a small one's), as the scratch allows (39 at
    // d = 32, K = 16), each of at least 32 tiles, one scan of every warp
    const int ES = na_entries(d);
    const int64_t tiles = (N + NA_P - 1) / NA_P;
    const int64_t want = (1216 + 2 * K - 1) / (2 * K), fit = (int64_t)(NA_SCRATCH / ((size_t)2 * K * ES));
    NaArgs a;
    a.X = X;
    a.N = N;
    a.d = d;
    a.z = z;
    a.zbar = zbar;
    a.K = K;
    a.G = (int)std::max<int64_t>(1, std::min(std::min(want, fit), (tiles + NA_Q * NA_W - 1) / (NA_Q * NA_W)));
    // as many FP32 groups as 256 threads hold 4 x 4 register blocks of the padded triangle
    StatLayout L;
    L.init(d, STAT_FULL);
    a.W = std::max(1, 256 / L.nblk);
    a.scratch = scratch;
    // launched with cudaLaunchKernel, whose return value is this launch's own error (an
    // error left behind by an unrelated earlier launch is neither reported nor cleared)
    const void* fn = d <= 4 ? (const void*)na_partial_kernel<3>
                   : d <= 8 ? (const void*)na_partial_kernel<5>
                   : d <= 16 ? (const void*)na_partial_kernel<9> : (const void*)na_partial_kernel<17>;
    void* a1[] = {(void*)&a};
    if (cudaLaunchKernel(fn, dim3(2 * K, a.G), dim3(32 * NA_W), a1, 0, s) != cudaSuccess) return DPMM_ECUDA;
    const double* cs = scratch;
    void* a2[] = {(void*)&d, (void*)&a.G, (void*)&K, (void*)&cs, (void*)&n_out, (void*)&sx_out, (void*)&sxx_out};
    if (cudaLaunchKernel((const void*)na_combine_kernel, dim3(2 * K, (ES + 31) / 32), dim3(256), a2, 0, s) != cudaSuccess)
        return DPMM_ECUDA;
    return DPMM_OK;
}
