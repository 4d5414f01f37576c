// xy_sf.cu -- structure factors S_par(k), S_perp(k) of the rotor lattice for
// the correlation-length extraction of arXiv 2409.06412, App. C.
//
// With rotors s = (cos(r theta), sin(r theta)) (the paper's definition is
// r = 1) on an N_par x N_perp lattice (x along the dimer rows, y across),
// Eq. S-as-lattice-FT reads
//   S_perp(k) = 1 / (N_perp N_par^2) sum_l sum_kappa |s~^kappa_{k,l}|^2,
// s~ the 2-D DFT of one rotor component.  Summing |.|^2 over l is, by
// Parseval, N_par times the sum over columns x of the 1-D DFT along y:
//   S_perp(k) = 1 / (N_perp N_par) sum_x sum_kappa |sum_y s^kappa_{x,y} e^{-2 pi i k y / N_perp}|^2,
// and likewise S_par(k) from the 1-D DFTs of the rows along x.  Only the
// wavenumbers k < K near the peak at k = 0 (Eq. Lorentzian-Peak) are formed: no
// 2-D transform is needed.
//
// Each line of N = R A sites is split once (Cooley and Tukey 1965; only the
// outputs k < K are formed in the second step):
//   X_k = sum_{a < A} w_N^{k a} Y_{k mod R}(a),  Y_j(a) = sum_{b < R} w_R^{j b} s_{a + A b},
// w_N = e^{-2 pi i / N}, with R the largest of 16, 8, 4, 2, 1 that divides N.
// The R-point transforms are real, so Y_{R - j} = conj Y_j and 62 additions and
// products serve 16 sites; cosine and sine rotor are the two halves of packed
// pairs.  That is 4 + 0.25 K packed instructions per site and direction at R = 16
// where the direct sums took 4 K scalar ones, and a shorter sum rounds less.  What
// bounds the kernels now is the accurate sine and cosine of every site (once per
// direction and 16 wavenumbers).  16 lattices of 1024^2, K = 16: 0.47 ms -> 0.12 ms a
// call (0.69 -> 0.17 ms when nothing else is in flight: no allocations per call).
//
// Line sums are FP32; the squared moduli are summed in FP64 per block and the
// blocks of a lattice in a fixed order by sf_finish_kernel (deterministic).
#include <algorithm>

#include "xy_device.cuh"

namespace xy {

namespace {

constexpr int kKC = 16;           // wavenumbers per pass
constexpr int kRowsPerBlock = 32;  // 8 warps of 4 rows, 8 lanes per row
constexpr int kColsPerBlock = 32;  // one per lane; the 8 warps share the column's sites
constexpr unsigned kFullS = 0xFFFFFFFFu;

// twiddles W[m] = (cos 2 pi m / N, sin 2 pi m / N), m < N
__device__ void build_twiddles(float2* W, int N)
{
    for (int m = threadIdx.x; m < N; m += blockDim.x) {
        float s, c;
        sincospif(2.0f * (float)m / (float)N, &s, &c);
        W[m] = make_float2(c, s);
    }
    __syncthreads();
}

__device__ __forceinline__ float2 neg2(float2 v) { return make_float2(-v.x, -v.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float k, float2 a) { return __fmul2_rn(splat2(k), a); }
__device__ __forceinline__ float2 fma2(float k, float2 a, float2 b) { return __ffma2_rn(splat2(k), a, b); }

// Y_j = sum_b z_b e^{-2 pi i j b / R}, j = 0 .. R / 2, of R real values (each a
// pair of independent ones).
template <int R>
__device__ __forceinline__ void dft_real(const float2 (&z)[R], float2 (&yr)[R / 2 + 1], float2 (&yi)[R / 2 + 1])
{
    const float h = 0.70710678118654752f;  // cos(pi / 4)
    const float2 zero = make_float2(0.f, 0.f);
    if constexpr (R == 1) {
        yr[0] = z[0];
        yi[0] = zero;
    } else if constexpr (R == 2) {
        yr[0] = add2(z[0], z[1]);
        yr[1] = sub2(z[0], z[1]);
        yi[0] = yi[1] = zero;
    } else if constexpr (R == 4) {
        const float2 a = add2(z[0], z[2]), b = add2(z[1], z[3]);
        yr[0] = add2(a, b);
        yr[2] = sub2(a, b);
        yr[1] = sub2(z[0], z[2]);
        yi[1] = sub2(z[3], z[1]);
        yi[0] = yi[2] = zero;
    } else {
        // halves: sums give the even outputs, differences the odd ones
        float2 e[R / 2], o[R / 2], er[R / 4 + 1], ei[R / 4 + 1];
#pragma unroll
        for (int i = 0; i < R / 2; ++i) {
            e[i] = add2(z[i], z[i + R / 2]);
            o[i] = sub2(z[i], z[i + R / 2]);
        }
        dft_real<R / 2>(e, er, ei);
#pragma unroll
        for (int j = 0; j <= R / 4; ++j) {
            yr[2 * j] = er[j];
            yi[2 * j] = ei[j];
        }
        if constexpr (R == 8) {
            const float2 d = sub2(o[1], o[3]), s = add2(o[1], o[3]);
            yr[1] = fma2(h, d, o[0]);
            yr[3] = fma2(-h, d, o[0]);
            yi[1] = fma2(-h, s, neg2(o[2]));
            yi[3] = fma2(-h, s, o[2]);
        } else {  // R == 16: terms i and 8 - i of the differences share their cosine and sine
            const float c1 = 0.92387953251128676f, c3 = 0.38268343236508977f;  // cos(pi / 8), cos(3 pi / 8)
            const float2 p1 = sub2(o[1], o[7]), p2 = sub2(o[2], o[6]), p3 = sub2(o[3], o[5]);
            const float2 q1 = add2(o[1], o[7]), q2 = add2(o[2], o[6]), q3 = add2(o[3], o[5]);
            const float2 A = fma2(h, p2, o[0]), B = fma2(-h, p2, o[0]);
            const float2 T1 = fma2(c3, p3, mul2(c1, p1)), T3 = fma2(-c1, p3, mul2(c3, p1));
            const float2 U = fma2(h, q2, o[4]), V = fma2(h, q2, neg2(o[4]));
            const float2 V1 = fma2(c1, q3, mul2(c3, q1)), V3 = fma2(-c3, q3, mul2(c1, q1));
            yr[1] = add2(A, T1);
            yr[7] = sub2(A, T1);
            yr[3] = add2(B, T3);
            yr[5] = sub2(B, T3);
            yi[1] = neg2(add2(U, V1));
            yi[7] = sub2(U, V1);
            yi[3] = neg2(add2(V, V3));
            yi[5] = sub2(V, V3);
        }
    }
}

// Adds the terms of one a to the sums X_k, k = k0 + q < K: p points at site a of
// the line, its sites a + A b are `stride` apart.
template <int R>
__device__ __forceinline__ void add_terms(const float* p, int64_t stride, float r, const float2* W, int N, int a, int k0,
                                          float2 (&xr)[kKC], float2 (&xi)[kKC])
{
    float t[R];
#pragma unroll
    for (int b = 0; b < R; ++b) t[b] = p[b * stride];
    float2 z[R], yr[R / 2 + 1], yi[R / 2 + 1];
#pragma unroll
    for (int b = 0; b < R; ++b) sincosf(r * t[b], &z[b].y, &z[b].x);
    dft_real<R>(z, yr, yi);
    int m = (int)(((int64_t)k0 * a) % N);  // k a mod N
#pragma unroll
    for (int q = 0; q < kKC; ++q) {
        const float2 w = W[m];  // w_N^{k a} = (w.x, -w.y)
        m += a;
        if (m >= N) m -= N;
        constexpr int half = R / 2;
        const int j = q % R;  // k0 is a multiple of 16, so of R
        const bool up = j > half;
        const int jj = up ? R - j : j;
        // X_k += (w.x - i w.y) (Y_re + i Y_im), Y_{R - j} = conj Y_j; the ends of the
        // half spectrum are real
        xr[q] = fma2(w.x, yr[jj], xr[q]);
        xi[q] = fma2(-w.y, yr[jj], xi[q]);
        if (jj != 0 && 2 * jj != R) {
            xr[q] = fma2(up ? -w.y : w.y, yi[jj], xr[q]);
            xi[q] = fma2(up ? -w.x : w.x, yi[jj], xi[q]);
        }
    }
}

__device__ __forceinline__ int radix_of(int N) { return N % 16 == 0 ? 16 : (N % 8 == 0 ? 8 : (N % 4 == 0 ? 4 : (N % 2 == 0 ? 2 : 1))); }

// The sums X_k of a line whose first site is p, sites `step` apart: the terms
// a = a0, a0 + da, ...
template <int R>
__device__ void line_sums(const float* p, int64_t step, float r, const float2* W, int N, int a0, int da, int k0,
                          float2 (&xr)[kKC], float2 (&xi)[kKC])
{
    const int A = N / R;
    for (int a = a0; a < A; a += da) add_terms<R>(p + a * step, A * step, r, W, N, a, k0, xr, xi);
}
__device__ __forceinline__ void line_sums_any(const float* p, int64_t step, float r, const float2* W, int N, int a0, int da,
                                              int k0, float2 (&xr)[kKC], float2 (&xi)[kKC])
{
    switch (radix_of(N)) {  // the same for the whole block
    case 16: line_sums<16>(p, step, r, W, N, a0, da, k0, xr, xi); break;
    case 8: line_sums<8>(p, step, r, W, N, a0, da, k0, xr, xi); break;
    case 4: line_sums<4>(p, step, r, W, N, a0, da, k0, xr, xi); break;
    case 2: line_sums<2>(p, step, r, W, N, a0, da, k0, xr, xi); break;
    default: line_sums<1>(p, step, r, W, N, a0, da, k0, xr, xi); break;
    }
}

__device__ __forceinline__ float2 shfl2(float2 v, int o)
{
    return make_float2(__shfl_xor_sync(kFullS, v.x, o), __shfl_xor_sync(kFullS, v.y, o));
}
__device__ __forceinline__ float norm2(float2 a, float2 b) { return a.x * a.x + a.y * a.y + b.x * b.x + b.y * b.y; }

}  // namespace

// S_par partials: block (lattice, row chunk, k chunk); 8 lanes per row take the
// terms a = l, l + 8, ...; part[((lat n_kc + kc) n_rc + rc) kKC + k - k0] = sum over
// the chunk's rows of sum_kappa |X_k|^2
__global__ void __launch_bounds__(256, 2) sf_rows_kernel(const float* theta, const SfLattice* lats, float r, double* part,
                                                         int n_rc)
{
    extern __shared__ float2 W[];
    const SfLattice lt = lats[blockIdx.x];
    const int rc = blockIdx.y, k0 = blockIdx.z * kKC;
    const int Lx = lt.Lx, Ly = lt.Ly;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (rc * kRowsPerBlock >= Ly) return;
    build_twiddles(W, Lx);
    const int l8 = lane & 7;
    const int y = rc * kRowsPerBlock + 4 * warp + (lane >> 3);
    float2 xr[kKC], xi[kKC];
#pragma unroll
    for (int q = 0; q < kKC; ++q) xr[q] = xi[q] = make_float2(0.f, 0.f);
    if (y < Ly) line_sums_any(theta + lt.offset + (int64_t)y * Lx, 1, r, W, Lx, l8, 8, k0, xr, xi);
    __syncwarp();
    // reduce-scatter over the row's 8 lanes: afterwards lane l holds the sums of
    // wavenumbers k0 + 2 l and k0 + 2 l + 1
#pragma unroll
    for (int o = 4, n = kKC / 2; o >= 1; o >>= 1, n >>= 1) {
        const bool hi = (l8 & o) != 0;
#pragma unroll
        for (int i = 0; i < kKC / 2; ++i)
            if (i < n) {
                const float2 sr = hi ? xr[i] : xr[i + n], si = hi ? xi[i] : xi[i + n];
                const float2 kr = hi ? xr[i + n] : xr[i], ki = hi ? xi[i + n] : xi[i];
                xr[i] = add2(kr, shfl2(sr, o));
                xi[i] = add2(ki, shfl2(si, o));
            }
    }
    // |X_k|^2 over the warp's four rows, then over the warps in order
    __shared__ double s_acc[8][kKC];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        double p = (double)norm2(xr[i], xi[i]);
        p += __shfl_xor_sync(kFullS, p, 8);
        p += __shfl_xor_sync(kFullS, p, 16);
        if (lane < 8) s_acc[warp][2 * lane + i] = p;
    }
    __syncthreads();
    if (threadIdx.x < kKC) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += s_acc[w][threadIdx.x];
        part[(((int64_t)blockIdx.x * gridDim.z + blockIdx.z) * n_rc + rc) * kKC + threadIdx.x] = t;
    }
}

// S_perp partials: block (lattice, 32 columns, k chunk); lane = column, warp w
// takes the terms a = w, w + 8, ... of it (one load of 32 consecutive sites per
// term), and the warps' sums are added in shared memory.
__global__ void __launch_bounds__(256, 2) sf_cols_kernel(const float* theta, const SfLattice* lats, float r, double* part,
                                                         int n_cc)
{
    extern __shared__ float2 W[];  // twiddles, later the sums [4 warps][2 kKC][32 columns]
    const SfLattice lt = lats[blockIdx.x];
    const int cc = blockIdx.y, k0 = blockIdx.z * kKC;
    const int Lx = lt.Lx, Ly = lt.Ly;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (cc * kColsPerBlock >= Lx) return;
    build_twiddles(W, Ly);
    const int x = cc * kColsPerBlock + lane;
    float2 xr[kKC], xi[kKC];
#pragma unroll
    for (int q = 0; q < kKC; ++q) xr[q] = xi[q] = make_float2(0.f, 0.f);
    if (x < Lx) line_sums_any(theta + lt.offset + x, Lx, r, W, Ly, warp, 8, k0, xr, xi);
    // tree over the warps: 4 + 4, 2 + 2, 1 + 1
    for (int h = 4; h >= 1; h >>= 1) {
        __syncthreads();  // the twiddles, or the last round's sums, have been read
        if (warp >= h && warp < 2 * h) {
#pragma unroll
            for (int q = 0; q < kKC; ++q) {
                W[((warp - h) * 2 * kKC + 2 * q) * 32 + lane] = xr[q];
                W[((warp - h) * 2 * kKC + 2 * q + 1) * 32 + lane] = xi[q];
            }
        }
        __syncthreads();
        if (warp < h) {
#pragma unroll
            for (int q = 0; q < kKC; ++q) {
                xr[q] = add2(xr[q], W[(warp * 2 * kKC + 2 * q) * 32 + lane]);
                xi[q] = add2(xi[q], W[(warp * 2 * kKC + 2 * q + 1) * 32 + lane]);
            }
        }
    }
    if (warp == 0) {
#pragma unroll
        for (int q = 0; q < kKC; ++q) {
            double p = (double)norm2(xr[q], xi[q]);
            for (int o = 16; o > 0; o >>= 1) p += __shfl_xor_sync(kFullS, p, o);
            if (lane == 0) part[(((int64_t)blockIdx.x * gridDim.z + blockIdx.z) * n_cc + cc) * kKC + q] = p;
        }
    }
}

// S[b][k] = (sum over the lattice's chunks of part) / (Lx Ly), k < K, of both directions
__global__ void sf_finish_kernel(const double* rows, const double* cols, const SfLattice* lats, int n_lat, int K, int n_kc,
                                 int n_rc, int n_cc, double* S_par, double* S_perp)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 2 * n_lat * K) return;
    const bool perp = i >= n_lat * K;
    const int bk = perp ? i - n_lat * K : i;
    const int b = bk / K, k = bk - b * K;
    const int n_chunks = perp ? n_cc : n_rc;
    const int mine = perp ? (lats[b].Lx + kColsPerBlock - 1) / kColsPerBlock : (lats[b].Ly + kRowsPerBlock - 1) / kRowsPerBlock;
    const double* p = (perp ? cols : rows) + ((int64_t)b * n_kc + k / kKC) * n_chunks * kKC + k % kKC;
    double t = 0.0;
    for (int c = 0; c < mine; ++c) t += p[(int64_t)c * kKC];
    (perp ? S_perp : S_par)[bk] = t / ((double)lats[b].Lx * (double)lats[b].Ly);
}

size_t sf_scratch_bytes(int n_lat, int max_x, int max_y, int K)
{
    const size_t n_kc = (size_t)(K + kKC - 1) / kKC;
    const size_t n_rc = (size_t)(max_y + kRowsPerBlock - 1) / kRowsPerBlock;
    const size_t n_cc = (size_t)(max_x + kColsPerBlock - 1) / kColsPerBlock;
    return sizeof(double) * (size_t)n_lat * n_kc * (n_rc + n_cc) * kKC;
}

cudaError_t launch_structure_factor(const float* theta, const SfLattice* lats, int n_lat, int max_x, int max_y, int K,
                                    float r, void* scratch, double* S_par, double* S_perp, int* n_launches,
                                    cudaStream_t st)
{
    if (n_lat == 0) return cudaSuccess;
    const int n_kc = (K + kKC - 1) / kKC;
    const int n_rc = (max_y + kRowsPerBlock - 1) / kRowsPerBlock;
    const int n_cc = (max_x + kColsPerBlock - 1) / kColsPerBlock;
    double* p_rows = static_cast<double*>(scratch);
    double* p_cols = p_rows + (size_t)n_lat * n_kc * n_rc * kKC;
    const size_t smem_x = max_x * sizeof(float2);
    const size_t smem_y = std::max(max_y * sizeof(float2), (size_t)4 * 2 * kKC * 32 * sizeof(float2));
    cudaError_t e = cudaSuccess;
    constexpr int smem_max = 8192 * (int)sizeof(float2);  // (the limit belongs to the kernel: always the largest)
    if (smem_x > 46 * 1024)
        e = cudaFuncSetAttribute(sf_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
    if (e == cudaSuccess && smem_y > 46 * 1024)
        e = cudaFuncSetAttribute(sf_cols_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
    if (e != cudaSuccess) return e;
    sf_rows_kernel<<<dim3((unsigned)n_lat, (unsigned)n_rc, (unsigned)n_kc), 256, smem_x, st>>>(theta, lats, r, p_rows, n_rc);
    sf_cols_kernel<<<dim3((unsigned)n_lat, (unsigned)n_cc, (unsigned)n_kc), 256, smem_y, st>>>(theta, lats, r, p_cols, n_cc);
    const int nt = 2 * n_lat * K;
    sf_finish_kernel<<<(nt + 255) / 256, 256, 0, st>>>(p_rows, p_cols, lats, n_lat, K, n_kc, n_rc, n_cc, S_par, S_perp);
    *n_launches += 3;
    return cudaGetLastError();
}

}  // namespace xy
