// xy_tau.cu -- integrated autocorrelation time and error of the mean of
// recorded observable series (arXiv 2409.06412, App. B: Eq.
// Autocorrelation-Function, Eq. Autocorrelation-Time, Eq. Time-Series-Var).
//
// For one series f_0 .. f_{n-1} (one lattice's records):
//   C(m)   = 1/(n - m) sum_s (f_s - f_bar)(f_{s+m} - f_bar),  C(0) = sigma_f^2
//   tau(M) = 1/2 + sum_{m=1}^{M} C(m) / C(0)                   (record units)
//   tau_C  = tau(M) at the smallest M >= 1 with M >= c tau(M) (the
//            self-consistent window), or at M = floor(n/2) (the paper's
//            tau_s / 2 taken literally) when half_window is set
//   sigma_mean = sqrt(2 tau_C sigma_f^2 / n)
// The mean and C(0) are FP64; the lag sums multiply FP32 deviations (relative
// 1e-7) and add runs of at most 256 terms into FP64.  Lags are formed 256 at a
// time and the window is checked after each batch, so a series with a short
// autocorrelation time costs one batch.
//
// A cluster of P blocks takes a series, each block an equal share of the sum over
// s, so that few series still fill the chip.  What bounds it: multiply-adds and
// the shared-memory reads that feed them, and the FP64 of the mean and C(0) (FP64
// issues at 1/64 of the FP32 rate).  A thread forms four lags of four sites from
// one aligned 16-byte read of its window and one that the warp shares: 16
// multiply-adds for two reads, where one lag per thread took two reads for each.
// The deviations of a series of up to kFullMax records stay in shared memory (a
// whole copy in each block, gathered from the cluster's other blocks); longer
// ones go through a global buffer and shared-memory tiles.  256 series of 10^4
// records, two batches: 0.94-1.14 ms -> 0.18 ms (0.10 ms of it multiply-adds, their
// reads and FP64 at the chip's rates; the rest is the barriers of the cluster).
#include <algorithm>

#include <cooperative_groups.h>

#include "xy_device.cuh"

namespace cg = cooperative_groups;

namespace xy {

namespace {

constexpr int kThreads = 256;
constexpr int kLags = 256;              // lags per batch
constexpr int kPad = kLags + 8;         // zeros past the last deviation that the windows read
constexpr int kFullMax = 48 * 1024;     // records whose deviations fit a block's shared memory
constexpr int kTile = 4096;             // sites per tile of a longer series
constexpr int kRun = 256;               // terms of one FP32 run

__device__ __forceinline__ double transform_value(double v, int transform)
{
    switch (transform) {
    case 1: return v * v;
    case 2: return (v * v) * (v * v);
    case 3: return fabs(v);
    default: return v;
    }
}

__device__ double block_sum(double v, double* s_red)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) s_red[warp] = v;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < kThreads / 32; ++w) t += s_red[w];
    return t;
}

// The sum of v over the cluster's threads, in rank order.
__device__ double cluster_sum(cg::cluster_group& cl, double v, double* s_red, double* s_one)
{
    v = block_sum(v, s_red);
    if (threadIdx.x == 0) *s_one = v;
    cl.sync();
    double t = 0.0;
    for (int r = 0; r < (int)cl.num_blocks(); ++r) t += *cl.map_shared_rank(s_one, r);
    cl.sync();  // s_one is read before it is written again
    return t;
}

// acc[i] += sum_{s < len} A[s] B[s + 4 g + i], i < 4: A, B 16-byte aligned, len a
// multiple of 4, B readable up to len + 4 g + 8
__device__ __forceinline__ void lag_sums(const float* A, const float* B, int len, int g, double (&acc)[4])
{
    const float4* a4 = reinterpret_cast<const float4*>(A);
    const float4* b4 = reinterpret_cast<const float4*>(B) + g;
    float4 w0 = b4[0];
    for (int s0 = 0; s0 < len; s0 += kRun) {
        const int s1 = min(len, s0 + kRun);
        float c0 = 0.f, c1 = 0.f, c2 = 0.f, c3 = 0.f;
#pragma unroll 4
        for (int s = s0; s < s1; s += 4) {
            const float4 a = a4[s >> 2];
            const float4 w1 = b4[(s >> 2) + 1];
            c0 = fmaf(a.x, w0.x, c0);
            c1 = fmaf(a.x, w0.y, c1);
            c2 = fmaf(a.x, w0.z, c2);
            c3 = fmaf(a.x, w0.w, c3);
            c0 = fmaf(a.y, w0.y, c0);
            c1 = fmaf(a.y, w0.z, c1);
            c2 = fmaf(a.y, w0.w, c2);
            c3 = fmaf(a.y, w1.x, c3);
            c0 = fmaf(a.z, w0.z, c0);
            c1 = fmaf(a.z, w0.w, c1);
            c2 = fmaf(a.z, w1.x, c2);
            c3 = fmaf(a.z, w1.y, c3);
            c0 = fmaf(a.w, w0.w, c0);
            c1 = fmaf(a.w, w1.x, c1);
            c2 = fmaf(a.w, w1.y, c2);
            c3 = fmaf(a.w, w1.z, c3);
            w0 = w1;
        }
        acc[0] += (double)c0;
        acc[1] += (double)c1;
        acc[2] += (double)c2;
        acc[3] += (double)c3;
    }
}

}  // namespace

// FULL: the series' deviations are whole in shared memory; else in `scratch`
// (n floats per series).
template <bool FULL>
__global__ void __launch_bounds__(kThreads) autocorr_kernel(const double2* rec, int64_t R, int component, int transform,
                                                            int64_t skip, int n, float* scratch, double c_win,
                                                            int half_window, double* out)
{
    extern __shared__ float4 s_dyn[];
    float* s_d = reinterpret_cast<float*>(s_dyn);  // FULL: the series; else a tile of s and its window
    __shared__ double s_red[kThreads / 32];
    __shared__ double s_one;
    __shared__ double s_C[4][kLags];  // the quarters' sums; [0] the block's
    __shared__ double s_tau;
    __shared__ int s_done;
    cg::cluster_group cl = cg::this_cluster();
    const int P = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int b = blockIdx.x / P;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double2* series = rec + (int64_t)b * R + skip;
    float* d = FULL ? s_d : scratch + (int64_t)b * n;
    // this block's share of the records, in multiples of four
    const int share = (int)((((int64_t)n + P - 1) / P + 3) / 4 * 4);
    const int lo = (int)min((int64_t)n, (int64_t)rank * share), hi = (int)min((int64_t)n, (int64_t)lo + share);
    if (tid == 0) s_done = 0;
    double acc = 0.0;
    for (int s = lo + tid; s < hi; s += kThreads) {
        const double2 r = series[s];
        acc += transform_value(component ? r.y : r.x, transform);
    }
    const double mean = cluster_sum(cl, acc, s_red, &s_one) / n;
    acc = 0.0;
    for (int s = lo + tid; s < hi; s += kThreads) {
        const double2 r = series[s];
        const double dv = transform_value(component ? r.y : r.x, transform) - mean;
        d[s] = (float)dv;
        acc += dv * dv;
    }
    // zeros behind the last deviation: a term that reaches past the series vanishes
    if (FULL)
        for (int s = n + tid; s < (n + 3) / 4 * 4 + kPad; s += kThreads) s_d[s] = 0.f;
    if (!FULL) __threadfence();  // the shares are read by the cluster's other blocks
    const double C0 = cluster_sum(cl, acc, s_red, &s_one) / n;  // also orders the writes of d before the lag sums
    if (FULL && P > 1) {  // the other blocks' shares
        for (int r = 0; r < P; ++r) {
            if (r == rank) continue;
            const float* o = cl.map_shared_rank(s_d, r);
            const int a = (int)min((int64_t)n, (int64_t)r * share), e = (int)min((int64_t)n, (int64_t)a + share);
            for (int s = a + tid; s < e; s += kThreads) s_d[s] = o[s];
        }
        cl.sync();  // and nobody leaves or goes on before its share has been read
    }
    const int M_max = n / 2;
    double tau = 0.5;  // of every thread of block 0
    bool done = !(C0 > 0.0);  // the same in every block
    // lags m0 .. m0 + 255 (lag 0 is formed and ignored): thread (g, quarter) takes
    // lags m0 + 4 g .. + 3 over a quarter of the block's share of s < n - m0
    const int g = tid & 63, quarter = tid >> 6;
    for (int m0 = 0; m0 <= M_max && !done; m0 += kLags) {
        double c4[4] = {0.0, 0.0, 0.0, 0.0};
        const int len = n - m0;
        const int part = (int)((((int64_t)len + P - 1) / P + 15) / 16 * 16);  // per block
        const int a0 = (int)min((int64_t)len, (int64_t)rank * part), a1 = (int)min((int64_t)len, (int64_t)a0 + part);
        if (FULL) {
            const int q0 = a0 + quarter * (part / 4), q1 = min((a1 + 3) / 4 * 4, q0 + part / 4);
            if (q0 < q1) lag_sums(s_d + q0, s_d + q0 + m0, q1 - q0, g, c4);
        } else {
            float* s_w = s_d + kTile;
            for (int t0 = a0; t0 < a1; t0 += kTile) {
                const int t1 = min(a1, t0 + kTile);
                __syncthreads();
                for (int s = tid; s < kTile; s += kThreads) s_d[s] = t0 + s < t1 ? d[t0 + s] : 0.f;
                for (int s = tid; s < kTile + kPad; s += kThreads) {
                    const int64_t w = (int64_t)t0 + m0 + s;
                    s_w[s] = w < n ? d[w] : 0.f;
                }
                __syncthreads();
                lag_sums(s_d + quarter * (kTile / 4), s_w + quarter * (kTile / 4), kTile / 4, g, c4);
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; ++i) s_C[quarter][4 * g + i] = c4[i];
        __syncthreads();
        s_C[0][tid] = (s_C[0][tid] + s_C[1][tid]) + (s_C[2][tid] + s_C[3][tid]);
        cl.sync();
        if (rank == 0) {
            const int m = m0 + tid;
            const bool in = m >= 1 && m <= M_max;
            double v = 0.0;
            if (in) {
                for (int r = 0; r < P; ++r) v += cl.map_shared_rank(&s_C[0][0], r)[tid];
                v = v / (double)(n - m) / C0;
            }
            // tau(m): inclusive sums over the lags, in the warp and then over the warps
            for (int o = 1; o < 32; o <<= 1) {
                const double u = __shfl_up_sync(0xFFFFFFFFu, v, o);
                if (lane >= o) v += u;
            }
            if (lane == 31) s_red[warp] = v;
            __syncthreads();
            double before = tau;
            for (int w = 0; w < warp; ++w) before += s_red[w];
            double total = tau;
            for (int w = 0; w < kThreads / 32; ++w) total += s_red[w];
            v += before;  // tau(m)
            const bool stop = in && (m == M_max || (!half_window && (double)m >= c_win * v));
            // the first lag that stops
            const unsigned hit = __ballot_sync(0xFFFFFFFFu, stop);
            __shared__ int s_hit[kThreads / 32];
            if (lane == 0) s_hit[warp] = hit ? __ffs(hit) - 1 + 32 * warp : kThreads;
            __syncthreads();
            int first = kThreads;
            for (int w = 0; w < kThreads / 32; ++w) first = min(first, s_hit[w]);
            if (tid == first) {
                s_tau = v;
                s_done = 1;
            }
            __syncthreads();
            tau = first < kThreads ? s_tau : total;
        }
        cl.sync();  // s_done for every block; s_C has been read
        done = *cl.map_shared_rank(&s_done, 0) != 0;
    }
    if (rank == 0 && tid == 0) {
        out[4 * b + 0] = mean;
        out[4 * b + 1] = C0;
        out[4 * b + 2] = tau;
        out[4 * b + 3] = sqrt(2.0 * tau * C0 / n);
    }
    cl.sync();  // block 0's s_done and every s_C stay until the last read of them
}

cudaError_t launch_autocorr(const double2* rec, int64_t n_series, int64_t R, int component, int transform,
                            int64_t skip, int n, double c_win, int half_window, double* out, cudaStream_t st)
{
    if (n_series == 0) return cudaSuccess;
    int dev = 0, sms = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // blocks per series: enough for about six per SM, each with at least 1024 records
    int P = 1;
    while (P < 8 && n_series * P < 6 * (int64_t)sms && n / (2 * P) >= 1024) P *= 2;
    const bool full = n <= kFullMax;
    const size_t smem = sizeof(float) * (full ? (size_t)(n + 3) / 4 * 4 + kPad : (size_t)2 * kTile + kPad);
    float* scratch = nullptr;
    cudaError_t e = cudaSuccess;
    const auto kern = full ? autocorr_kernel<true> : autocorr_kernel<false>;
    // (the limit belongs to the kernel, which other calls share: always the largest)
    if (smem > 32 * 1024)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(sizeof(float) * (full ? kFullMax + kPad : 2 * kTile + kPad)));
    if (e == cudaSuccess && !full)
        e = cudaMallocAsync(&scratch, sizeof(float) * (size_t)n_series * n, st);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)(n_series * P));
    lc.blockDim = dim3(kThreads);
    lc.dynamicSmemBytes = smem;
    lc.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)P;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    e = cudaLaunchKernelEx(&lc, kern, rec, R, component, transform, skip, n, scratch, c_win, half_window, out);
    if (scratch) cudaFreeAsync(scratch, st);
    return e;
}

}  // namespace xy
