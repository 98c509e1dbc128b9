// Double-loop (nested) Monte Carlo estimate of the expected information gain, the
// direct sampling of Eq. expected_I that the Laplace method of Thm 4 replaces
// (Sec. 4.4 compares the two).  With y_n = g(theta_n) + eps_n and Gaussian noise
// C_eps = sigma^2 I,
//   log_ev[n] = log( (1/M) sum_m exp(-|y_n - g(theta'_m)|^2 / (2 sigma^2)) )
//   I_DL      = (1/N) sum_n [ -|eps_n|^2 / (2 sigma^2) - log_ev[n] ]
// (the normalising constant of the Gaussian likelihood cancels).  The sums are FP64, of squared
// distances summed from the differences themselves (no |y|^2 + |g|^2 - 2 y.g expansion, which
// cancels catastrophically when the noise is small).
//
// FP64 runs 64 times slower than FP32 here, and only the inner samples near a row's best
// contribute to its log-sum-exp: k_screen computes every distance in FP32 (of values scaled
// by 1 / (sigma sqrt 2), so a distance is -l), and k_log_evidence computes in FP64 those that
// can matter.  A pair (n, m) is left out only when a rigorous lower bound of its distance,
// from its FP32 value, exceeds an upper bound of the row's smallest by
// (kDropBits + log2 M) ln 2: all left-out terms together are then below 2^-kDropBits of the
// sum's largest term, far below the rounding of the sum.  With u = 2^-24, rounding the scaled
// inputs moves a distance's root by at most eta = u (|y_n| + max_m |g_m|) (and 1e-22 where
// they underflow), the FP32 sum of squares its value by a factor within 1 +- (D + 8) u.
// Values that FP32 cannot hold (overflow, NaN) are always kept.
//
// Both sides measured (N = M = 4096, sigma = 0.01, the paper's study): D = 204, where 1.3% of the
// pairs are kept, 17.8 ms with every pair in FP64 (two FP64 operations a pair and entry, tiles of
// 32 x 64) and 0.72 ms screened (0.30 the FP32 distances, 0.40 the FP64 part), both 3e-16 from 64 bits;
// D = 72, records that end before the waves arrive and every pair matters, 8.0 and 5.2 ms.
#include <math.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "dlmc_groups.h"
#include "oed_internal.cuh"

namespace oed {

constexpr int kSN = kScreenRows, kSM = 64, kSD = 32;      // k_screen: block tile and chunk of the data dimension
constexpr int kDropBits = 60;

// y_n = g_outer[n] + eps[n], scaled and rounded to FP32; g likewise
__device__ __forceinline__ float screen_value(double v, double scale) { return (float)(v * scale); }

// The screened values, rows padded with zeros to Dp entries: y of the rows below N, -g of the
// next M rows (a sum is then the difference), and max_m |g_m| as the bits of a float (rounded
// up).  One warp per row.
__global__ void __launch_bounds__(256) k_screen_values(const double *__restrict__ g_out, const double *__restrict__ eps,
                                                       int N, const double *__restrict__ g_in, int M, int D, int Dp,
                                                       double scale, float *__restrict__ val, unsigned *__restrict__ gmax)
{
    const size_t r = (size_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (r >= (size_t)N + M) return;
    float s = 0.0f;
    for (int d = lane; d < Dp; d += 32) {
        float v = 0.0f;
        if (d < D) v = r < N ? screen_value(g_out[r * D + d] + eps[r * D + d], scale)
                             : -screen_value(g_in[(r - N) * D + d], scale);
        val[r * Dp + d] = v;
        s = fmaf(v, v, s);
    }
    if (r < N) return;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    // the sum's rounding is within (D + 8) u as above; NaN and overflow raise the bound to infinity
    const float q = sqrtf(s) * (1.0f + (D + 8) * 6e-8f);
    if (lane == 0) atomicMax(gmax, __float_as_uint(q <= 3e38f ? q : INFINITY));
}

// dist[n - n0][m] = |y_n - g_m|^2 in FP32 for the rows n0 .. n1 - 1, and per row the bits of the
// smallest (finite) one.  A thread owns a 4 x 4 tile and two data entries at a time (.f32x2).
__global__ void __launch_bounds__(256) k_screen(const float *__restrict__ val, int N, int n0, int n1, int M, int Dp,
                                                float *__restrict__ dist, unsigned *__restrict__ best)
{
    __shared__ float2 ys[kSD / 2][kSN + 1], gs[kSD / 2][kSM + 1];
    const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
    const int nb = n0 + blockIdx.y * kSN, mb = blockIdx.x * kSM;
    const float *gval = val + (size_t)N * Dp;
    float2 acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] = make_float2(0.0f, 0.0f);
    for (int d0 = 0; d0 < Dp; d0 += kSD) {
#pragma unroll
        for (int q = 0; q < kSN * kSD / 256; q++) {
            const int k = tid + 256 * q, r = k / kSD, c = k % kSD;
            const float y = nb + r < n1 ? val[(size_t)(nb + r) * Dp + d0 + c] : 0.0f;
            const float g = mb + r < M ? gval[(size_t)(mb + r) * Dp + d0 + c] : 0.0f;
            (&ys[c >> 1][r].x)[c & 1] = y;
            (&gs[c >> 1][r].x)[c & 1] = g;
        }
        __syncthreads();
#pragma unroll 4
        for (int c = 0; c < kSD / 2; c++) {
            float2 y[4], g[4];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                y[i] = ys[c][ty + 16 * i];
                g[i] = gs[c][tx + 16 * i];
            }
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const float2 e = __fadd2_rn(y[i], g[j]);
                    acc[i][j] = __ffma2_rn(e, e, acc[i][j]);
                }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const int n = nb + ty + 16 * i;
        float b = INFINITY;
        if (n < n1)
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int m = mb + tx + 16 * j;
                if (m >= M) continue;
                const float v = acc[i][j].x + acc[i][j].y;
                dist[(size_t)(n - n0) * M + m] = v;
                b = fminf(b, v);   // ignores NaN
            }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) b = fminf(b, __shfl_xor_sync(0xffffffffu, b, o));
        if (tx == 0 && n < n1) atomicMin(best + n, __float_as_uint(b));
    }
}

// log_ev[n], one block per row: collect the samples to keep, 32 at a time and a lane each, sum
// their squared differences in FP64 in the order of the data, and fold them into a running
// (max, sum of exponentials) per lane; e2[n] = |eps_n|^2 where asked for.  dist NULL: all are kept.
constexpr int kEvWarps = 4, kEvPer = 8, kEvList = 2048;   // warps, samples a lane looks at per round, list
constexpr int kEvShared = 12288;   // longest data row kept in shared memory (96 KB)

// (max, sum) of a warp's lanes; every lane gets them.  A lane without a comparable distance holds
// (-inf, 0), or (-inf, NaN) after a distance that is NaN: its sum goes on as it is, so a NaN meets
// the samples of the other lanes and warps.
__device__ __forceinline__ void warp_log_sum(double &mx, double &sm)
{
    double top = mx;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) top = fmax(top, __shfl_xor_sync(0xffffffffu, top, o));
    double s = mx > -INFINITY ? sm * exp(mx - top) : sm;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    mx = top;
    sm = s;
}

template <bool SHARED>
__global__ void __launch_bounds__(32 * kEvWarps) k_log_evidence(
    const double *__restrict__ g_out, const double *__restrict__ eps, int n0, const double *__restrict__ g_in, int M, int D,
    int Dp, double inv2s2, double log_m, float slack, const float *__restrict__ val, const float *__restrict__ dist,
    const unsigned *__restrict__ best, const unsigned *__restrict__ gmax, int vec, double *__restrict__ log_ev,
    double *__restrict__ e2)
{
    extern __shared__ double ys[];   // [D] this row's data
    __shared__ int list[kEvList];
    __shared__ int wcount[kEvWarps];
    __shared__ double red[2][kEvWarps];
    __shared__ float rednorm[kEvWarps];
    const int n = n0 + blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float ynorm = 0.0f;
    double e = 0.0;
    for (unsigned d = tid; d < (unsigned)D; d += blockDim.x) {
        const double ep = eps[(size_t)n * D + d];
        if (SHARED) ys[d] = g_out[(size_t)n * D + d] + ep;
        e = fma(ep, ep, e);
        if (dist) {
            const float v = val[(size_t)n * Dp + d];
            ynorm = fmaf(v, v, ynorm);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ynorm += __shfl_xor_sync(0xffffffffu, ynorm, o);
        e += __shfl_xor_sync(0xffffffffu, e, o);
    }
    if (lane == 0) {
        red[0][warp] = e;
        rednorm[warp] = ynorm;
    }
    __syncthreads();
    float limit = INFINITY;   // keep distances up to this
    if (dist) {
        float y2 = 0.0f;
        for (int k = 0; k < kEvWarps; k++) y2 += rednorm[k];
        if (e2 && tid == 0) e2[n] = (red[0][0] + red[0][1]) + (red[0][2] + red[0][3]);
        // every operation rounds the limit up
        const float u = 5.9604644775390625e-08f, kappa = (D + 8) * u, up = __fadd_ru(1.0f, __fmul_ru(kappa, 1.001f));
        const float eta = __fadd_ru(__fmul_ru(__fmul_ru(u, 1.001f), __fadd_ru(__fmul_ru(__fsqrt_ru(y2), up),
                                                                             __uint_as_float(*gmax))), 1e-22f * D);
        const float lo = __fadd_ru(__fmul_ru(__fsqrt_ru(__uint_as_float(best[n])), up), eta);
        const float root = __fdiv_ru(__fadd_ru(__fsqrt_ru(__fadd_ru(__fmul_ru(lo, lo), slack)), eta),
                                     __fadd_rd(1.0f, -1.001f * kappa));
        const float lim = __fmul_ru(root, root);
        if (lim < 1e38f && kappa < 0.01f) limit = lim;
    }
    auto data = [&](int d) { return SHARED ? ys[d] : g_out[(size_t)n * D + d] + eps[(size_t)n * D + d]; };
    double mx = -INFINITY, sm = 0.0;
    const float *row = dist ? dist + (size_t)blockIdx.x * M : nullptr;
    for (unsigned m0 = 0; m0 < (unsigned)M;) {   // (unsigned: a round ends up to 1023 samples past M)
        // the next samples to keep, in order, up to a full list
        int have = 0;
        __syncthreads();
        while (m0 < (unsigned)M && have + kEvPer * (int)blockDim.x <= kEvList) {
            // a warp takes kEvPer x 32 consecutive samples; kept unless known to be above the
            // limit (NaN and overflow are kept)
            unsigned b[kEvPer];
            int mine = 0;
#pragma unroll
            for (int q = 0; q < kEvPer; q++) {
                const unsigned m = m0 + (warp * kEvPer + q) * 32 + lane;
                const float v = row && m < (unsigned)M ? row[m] : 0.0f;
                b[q] = __ballot_sync(0xffffffffu, m < (unsigned)M && (!(v > limit) || !(v < 3e38f)));
                mine += __popc(b[q]);
            }
            if (lane == 0) wcount[warp] = mine;
            __syncthreads();
            int at = have;
            for (int k = 0; k < kEvWarps; k++) {
                if (k < warp) at += wcount[k];
                have += wcount[k];
            }
#pragma unroll
            for (int q = 0; q < kEvPer; q++) {
                if (b[q] >> lane & 1) list[at + __popc(b[q] & ((1u << lane) - 1u))] = (int)(m0 + (warp * kEvPer + q) * 32 + lane);
                at += __popc(b[q]);
            }
            m0 += kEvPer * blockDim.x;
            __syncthreads();
        }
        for (int k = tid; k < have; k += blockDim.x) {
            const double *g = g_in + (size_t)list[k] * D;
            double acc = 0.0;
            int d = 0;
            if (vec)
#pragma unroll 4
                for (; d < D; d += 2) {
                    const double2 v = *reinterpret_cast<const double2 *>(g + d);
                    const double a0 = data(d) - v.x, a1 = data(d + 1) - v.y;
                    acc = fma(a0, a0, acc);
                    acc = fma(a1, a1, acc);
                }
            for (; d < D; d++) {
                const double a0 = data(d) - g[d];
                acc = fma(a0, a0, acc);
            }
            const double l = -acc * inv2s2;
            const double t = exp(-fabs(l - mx));
            if (l > mx) {
                sm = sm * t + 1.0;
                mx = l;
            } else if (!(l == -INFINITY)) {   // (an infinite distance adds nothing)
                sm += t;
            }
        }
    }
    // combine the lanes, then the warps
    if (__any_sync(0xffffffffu, mx > -INFINITY || sm != 0.0)) warp_log_sum(mx, sm);
    if (lane == 0) {
        red[0][warp] = mx;
        red[1][warp] = sm;
    }
    __syncthreads();
    if (warp == 0) {
        mx = lane < kEvWarps ? red[0][lane] : -INFINITY;
        sm = lane < kEvWarps ? red[1][lane] : 0.0;
        warp_log_sum(mx, sm);
        // (a row without one comparable distance: -inf)
        if (lane == 0) log_ev[n] = mx > -INFINITY ? mx + log(sm) - log_m : -INFINITY;
    }
}

// I_DL = (1/N) sum_n [-|eps_n|^2 inv2s2 - log_ev[n]]: one block, fixed summation order; e2 NULL:
// the squared norms of the noise are summed here
__global__ void __launch_bounds__(512) k_dlmc_sum(const double *__restrict__ eps, const double *__restrict__ e2,
                                                  const double *__restrict__ log_ev, int N, int D, double inv2s2,
                                                  double *__restrict__ eig)
{
    __shared__ double sv[512];
    const int t = threadIdx.x, T = blockDim.x;
    double v = 0.0;
    for (long long n = t; n < N; n += T) {
        double q = 0.0;
        if (e2)
            q = e2[n];
        else
            for (int d = 0; d < D; d++) q = fma(eps[(size_t)n * D + d], eps[(size_t)n * D + d], q);
        v += -q * inv2s2 - log_ev[n];
    }
    sv[t] = v;
    __syncthreads();
    for (int s = T / 2; s > 0; s >>= 1) {
        if (t < s) sv[t] += sv[t + s];
        __syncthreads();
    }
    if (t == 0) *eig = sv[0] / N;
}

// The calls' scratch comes from a memory pool of the library's own (one per device, for all threads
// and streams) that keeps up to kScratchKept bytes across synchronisation.  From the device's pool,
// which gives everything back, the mapping took each call after a synchronise 0.2 ms: N = M = 8, D =
// 16 240 us against 100 with no scratch and every pair in FP64.  oed_destroy gives back what is kept,
// and so does oed_create where memory is short.
constexpr int kMaxDevices = 64;
constexpr unsigned long long kScratchKept = 256ull << 20;
static std::mutex g_scratch_mu;
static cudaMemPool_t g_scratch[kMaxDevices];

static cudaError_t scratch_alloc(void **p, size_t bytes, cudaStream_t st)
{
    int dev = 0;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaStreamIsCapturing(st, &cap);
    if (e != cudaSuccess) return e;
    // (a graph owns the memory of its own allocations)
    if (cap != cudaStreamCaptureStatusNone || dev >= kMaxDevices) return cudaMallocAsync(p, bytes, st);
    cudaMemPool_t pool = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_scratch_mu);
        if (!g_scratch[dev]) {
            cudaMemPoolProps props = {};
            props.allocType = cudaMemAllocationTypePinned;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = dev;
            unsigned long long keep = kScratchKept;
            e = cudaMemPoolCreate(&pool, &props);
            if (e == cudaSuccess) e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
            if (e != cudaSuccess) {
                if (pool) cudaMemPoolDestroy(pool);
                return e;
            }
            g_scratch[dev] = pool;
        }
        pool = g_scratch[dev];
    }
    return cudaMallocFromPoolAsync(p, bytes, pool, st);
}

void scratch_trim()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev >= kMaxDevices) return;
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    if (g_scratch[dev] && cudaMemPoolTrimTo(g_scratch[dev], 0) != cudaSuccess)
        cudaGetLastError();   // (nothing for a later call to report)
}

}  // namespace oed

extern "C" int oed_dlmc(const double *g_outer, const double *eps, int N, const double *g_inner, int M, int D,
                        double sigma, double *log_ev, double *eig, void *stream)
{
    using namespace oed;
    if (N < 1 || M < 1 || D < 1 || !g_outer || !eps || !g_inner || !log_ev || !(sigma > 0.0))
        return OED_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    const double inv2s2 = 1.0 / (2.0 * sigma * sigma), scale = sqrt(inv2s2);
    // scratch: [N] |eps|^2, the screened values, the distances of a group of rows, [N] smallest
    // distances, the largest norm.  Without it (the device is full) every pair is kept, at more time.
    const int Dp = (D + kSD - 1) / kSD * kSD;
    const int rows = dlmc_group_rows(N, M);
    const size_t nval = ((size_t)N + M) * Dp, ndist = (size_t)rows * M;
    double *e2 = nullptr;
    if (scratch_alloc((void **)&e2, (size_t)N * 8 + (nval + ndist + N + 1) * 4, st) != cudaSuccess) {
        cudaGetLastError();
        e2 = nullptr;
    }
    float *val = e2 ? (float *)(e2 + N) : nullptr, *dist = e2 ? val + nval : nullptr;
    unsigned *best = e2 ? (unsigned *)(dist + ndist) : nullptr, *gmax = e2 ? best + N : nullptr;
    if (e2) {
        cudaMemsetAsync(best, 0x7f, (size_t)N * 4, st);
        cudaMemsetAsync(gmax, 0, 4, st);
        k_screen_values<<<(unsigned)(((size_t)N + M + 7) / 8), 256, 0, st>>>(g_outer, eps, N, g_inner, M, D, Dp, scale,
                                                                             val, gmax);
    }
    const int vec = D % 2 == 0 && (uintptr_t)g_inner % 16 == 0;
    const bool shared = D <= kEvShared;
    const double log_m = std::log((double)M);
    const float slack = (float)((kDropBits * 0.6931471805599453 + log_m) * 1.000001);
    if (shared)
        cudaFuncSetAttribute(k_log_evidence<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kEvShared * 8);
    dlmc_for_groups(N, M, [&](int n0, int n1) {
        if (dist)
            k_screen<<<dim3((M - 1) / kSM + 1, (n1 - n0 - 1) / kSN + 1), 256, 0, st>>>(val, N, n0, n1, M, Dp, dist,
                                                                                          best);
        if (shared)
            k_log_evidence<true><<<n1 - n0, 32 * kEvWarps, (size_t)D * 8, st>>>(
                g_outer, eps, n0, g_inner, M, D, Dp, inv2s2, log_m, slack, val, dist, best, gmax, vec, log_ev, e2);
        else
            k_log_evidence<false><<<n1 - n0, 32 * kEvWarps, 0, st>>>(
                g_outer, eps, n0, g_inner, M, D, Dp, inv2s2, log_m, slack, val, dist, best, gmax, vec, log_ev, e2);
    });
    if (eig) k_dlmc_sum<<<1, 512, 0, st>>>(eps, e2, log_ev, N, D, inv2s2, eig);
    if (e2) cudaFreeAsync(e2, st);
    return cudaGetLastError() == cudaSuccess ? OED_OK : OED_ECUDA;
}
