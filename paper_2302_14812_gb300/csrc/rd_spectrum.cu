// Power spectra of the detector's time series (Section 4: the detector data are Fourier
// transformed in time and compared with the synchrotron spectra, Eq. 8 and Eq. 9).
//
// For every cell j and frequency index k = 0..N/2 (N = n_bins, a power of two):
//     P[j][k] = dt_det^2 * sum_c | sum_b F_c[j][b] exp(-2 pi i k b / N) |^2
// with F = E or B.  Two complex transforms per cell carry the three real components:
// Z1 = F_x + i F_y gives |Fx(k)|^2 + |Fy(k)|^2 = (|Z1(k)|^2 + |Z1(N-k)|^2) / 2, and Z2 = F_z gives
// |Fz(k)|^2 = |Z2(k)|^2.  Twiddles exp(-2 pi i j / N) are computed in FP64 once per length.
// N <= kFusedMaxN: one kernel reads a cell's bins, runs both FP32 transforms through shared
// memory and writes the cell's spectrum (the fields are read once, the spectrum written once).
// Longer series, up to kSplitMaxN: N = N1 N2, two kernels that read and write each element once (transforms
// of length N1 over the columns, of length N2 over the rows).  Beyond that: FP32 Stockham radix-2 passes
// over the whole batch, one launch per pass.
#include <math.h>

#include <algorithm>

#include "rd_internal.cuh"

namespace rd {

namespace {

__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// Z[2 j][b] = F_x + i F_y,  Z[2 j + 1][b] = F_z + 0 i  (component offset c0 = 0 for E, 3 for B), from the fields of an
// RD_FP64 detector (an RD_MIXED one has no series this long)
__global__ void k_pack_spectrum_input(const double* __restrict__ fields, int n_pix, int n_bins, int c0,
                                      float2* __restrict__ z)
{
    const long long total = (long long)n_pix * n_bins;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const long long j = i / n_bins, b = i - j * n_bins;
        const double* f = fields + i * 6 + c0;
        z[(2 * j) * n_bins + b] = make_float2((float)f[0], (float)f[1]);
        z[(2 * j + 1) * n_bins + b] = make_float2((float)f[2], 0.f);
    }
}

// One Stockham pass (n = N / s, s = 2^stage) over `batch` transforms of length N:
//   a = x[q + s p], b = x[q + s (p + n/2)],  y[q + s 2p] = a + b,  y[q + s (2p + 1)] = (a - b) w^p,
// w = exp(-2 pi i / n), p < n/2, q < s; w^p = tw[p s] with tw[j] = exp(-2 pi i j / N).
__global__ void k_fft_pass(const float2* __restrict__ x, float2* __restrict__ y, int N, int s,
                           const float2* __restrict__ tw, long long batch)
{
    const int half = N >> 1;
    const long long total = batch * half;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const long long bt = t / half;
        const int i = (int)(t - bt * half);          // i = p s + q
        const int q = i & (s - 1);
        const int p = i / s;
        const float2* xb = x + bt * N;
        float2* yb = y + bt * N;
        const float2 a = xb[i], b = xb[i + half];
        const float2 w = tw[p * s];
        yb[q + 2 * s * p] = make_float2(a.x + b.x, a.y + b.y);
        yb[q + 2 * s * p + s] = cmul(make_float2(a.x - b.x, a.y - b.y), w);
    }
}

__global__ void k_spectrum_power(const float2* __restrict__ X, int n_pix, int N, float scale,
                                 float* __restrict__ P)
{
    const int nk = N / 2 + 1;
    const long long total = (long long)n_pix * nk;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const long long j = i / nk;
        const int k = (int)(i - j * nk);
        const int km = (N - k) & (N - 1);
        const float2 z1 = X[(2 * j) * N + k], z1m = X[(2 * j) * N + km], z2 = X[(2 * j + 1) * N + k];
        const float pxy = 0.5f * (z1.x * z1.x + z1.y * z1.y + z1m.x * z1m.x + z1m.y * z1m.y);
        const float pz = z2.x * z2.x + z2.y * z2.y;
        P[i] = scale * (pxy + pz);
    }
}

// The three components c0..c0+2 (E: c0 = 0, B: c0 = 3) of bin b of a cell's row, with vector loads.
template <typename T, int STRIDE>
struct Load3;
template <>
struct Load3<float, 8> {
    static __device__ __forceinline__ float3 get(const float* row, int b, int c0)
    {
        const float* v = row + (size_t)b * 8;
        const float4 a = __ldg(reinterpret_cast<const float4*>(v));
        if (c0 == 0) return make_float3(a.x, a.y, a.z);
        const float2 c = __ldg(reinterpret_cast<const float2*>(v + 4));
        return make_float3(a.w, c.x, c.y);
    }
};
template <>
struct Load3<double, 6> {
    static __device__ __forceinline__ float3 get(const double* row, int b, int c0)
    {
        const double* v = row + (size_t)b * 6;
        if (c0 == 0) {
            const double2 a = __ldg(reinterpret_cast<const double2*>(v));
            return make_float3((float)a.x, (float)a.y, (float)__ldg(v + 2));
        }
        const double2 c = __ldg(reinterpret_cast<const double2*>(v + 4));
        return make_float3((float)__ldg(v + 3), (float)c.x, (float)c.y);
    }
};

// Shared-memory index of element i of a transform: one float2 of padding after every 16, so that
// the strided reads and writes of every radix-16 pass (and of the shorter last pass) fall on
// distinct banks.
__device__ __forceinline__ int pad(int i) { return i + (i >> 4); }

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }

// a * exp(-2 pi i j / 16), j = 0..7 a compile-time constant after unrolling: the trivial roots (1, -i) without a
// multiply, the others to twice FP32's digits (hi + lo, both rounded from the exact values): the lo parts are added
// to the smaller product before its rounding, so only the two roundings of an exact root's product remain.
__device__ __forceinline__ float2 mul_root16(float2 a, int j)
{
    if (j == 0) return a;
    if (j == 4) return make_float2(a.y, -a.x);
    constexpr double c1 = 0.92387953251128674, s1 = 0.38268343236508978, h = 0.70710678118654752;
    if (j == 2 || j == 6) {             // (+-1 - i) / sqrt 2
        const float hh = (float)h, hl = (float)(h - (double)(float)h);
        const float u = a.x + a.y, v = a.y - a.x;
        const float hu = __fmaf_rn(u, hh, __fmul_rn(u, hl)), hv = __fmaf_rn(v, hh, __fmul_rn(v, hl));
        return j == 2 ? make_float2(hu, hv) : make_float2(hv, -hu);
    }
    constexpr double re[8] = {1., c1, h, s1, 0., -s1, -h, -c1}, im[8] = {0., -s1, -h, -c1, -1., -c1, -h, -s1};
    const float rh = (float)re[j], rl = (float)(re[j] - (double)rh);
    const float ih = (float)im[j], il = (float)(im[j] - (double)ih);
    const float x = __fmaf_rn(a.y, ih, __fmaf_rn(a.y, il, -__fmul_rn(a.x, rl)));
    const float y = __fmaf_rn(a.y, rh, __fmaf_rn(a.y, rl, __fmul_rn(a.x, il)));
    return make_float2(__fmaf_rn(a.x, rh, -x), __fmaf_rn(a.x, ih, y));
}

// In-register DFT of length R (2, 4, 8, 16): X[k] = sum_r a[r] exp(-2 pi i r k / R), by radix-2
// decimation in frequency; the result is left in bit-reversed order (a[bitrev(k)] = X[k]).
template <int R>
constexpr int log2_of() { return R == 16 ? 4 : R == 8 ? 3 : R == 4 ? 2 : 1; }

template <int R>
__device__ __forceinline__ void dft_bitrev(float2 (&a)[R])
{
    constexpr int L = log2_of<R>();
#pragma unroll
    for (int st = 0; st < L; ++st) {
        const int h = R >> (st + 1);                            // span of this stage
#pragma unroll
        for (int g = 0; g < (1 << st); ++g) {
#pragma unroll
            for (int i = 0; i < R / (2 << st); ++i) {
                const int j = g * (R >> st);
                const float2 u = a[j + i], v = a[j + i + h];
                a[j + i] = cadd(u, v);
                const float2 d = csub(u, v);                    // times exp(-2 pi i i / (2h))
                a[j + i + h] = mul_root16(d, i * (8 / h));
            }
        }
    }
}

template <int R>
__device__ __forceinline__ constexpr int bitrev(int k)
{
    constexpr int L = log2_of<R>();
    int r = 0;
#pragma unroll
    for (int i = 0; i < L; ++i) r |= ((k >> i) & 1) << (L - 1 - i);
    return r;
}

// exp(-2 pi i j / N) for 0 <= j < N from the half-circle table tw[j] (j < N/2, in shared memory)
__device__ __forceinline__ float2 twiddle(const float2* tw, int j, int half_n)
{
    if (j < half_n) return tw[j];
    const float2 w = tw[j - half_n];
    return make_float2(-w.x, -w.y);
}

// One Stockham pass of radix R on both transforms of a cell (in place in shared memory, or reading
// the cell's bins from global memory when s = 1 and G): with n = N / s and m = n / R, butterfly
// (p, q), p < m, q < s, takes a_r = x[q + s (p + r m)], r < R, forms b_k = DFT_R(a)[k] and writes
// y[q + s (R p + k)] = b_k exp(-2 pi i p k / n).  After the passes of radices R1 R2 ... = N the
// transform is in natural order.  Each thread holds 16 elements of each transform (16 / R
// butterflies); all reads of a pass finish before its writes.
template <int R, bool G, typename T, int STRIDE>
__device__ __forceinline__ void spec_pass(float2* z1, float2* z2, const T* row, int c0, int N, int s,
                                          const float2* tw, int tid)
{
    constexpr int NB = 16 / R;                  // butterflies per thread
    const int n = N / s, m = n / R;
    const int nb = N / R;                       // butterflies per transform
    float2 a1[NB][R], a2[NB][R];
    int bq[NB], bp[NB];
    bool on[NB];
#pragma unroll
    for (int u = 0; u < NB; ++u) {
        const int t = tid + u * blockDim.x;
        on[u] = t < nb;
        bq[u] = t % s;
        bp[u] = t / s;
        if (on[u]) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int i = bq[u] + s * (bp[u] + r * m);
                if (G) {
                    const float3 v = Load3<T, STRIDE>::get(row, i, c0);
                    a1[u][r] = make_float2(v.x, v.y);
                    a2[u][r] = make_float2(v.z, 0.f);
                } else {
                    a1[u][r] = z1[pad(i)];
                    a2[u][r] = z2[pad(i)];
                }
            }
        }
    }
    __syncthreads();    // every read of the pass is done (first pass: the twiddle table is filled)
    const int half_n = N >> 1;
#pragma unroll
    for (int u = 0; u < NB; ++u) {
        if (!on[u]) continue;
        dft_bitrev<R>(a1[u]);
        dft_bitrev<R>(a2[u]);
        const int o = bq[u] + s * R * bp[u];
#pragma unroll
        for (int k = 0; k < R; ++k) {
            float2 b1 = a1[u][bitrev<R>(k)], b2 = a2[u][bitrev<R>(k)];
            if (k > 0) {
                const float2 w = twiddle(tw, bp[u] * k * s, half_n);      // exp(-2 pi i p k / n)
                b1 = cmul(b1, w);
                b2 = cmul(b2, w);
            }
            z1[pad(o + s * k)] = b1;
            z2[pad(o + s * k)] = b2;
        }
    }
    __syncthreads();
}

// The passes after the first, at stride S, of a length-N transform: radix 16 while 16 elements
// remain per butterfly, then the remaining radix (a compile-time sequence, so that every pass's
// registers are allocated on their own).
template <int N, int S, typename T, int STRIDE>
__device__ __forceinline__ void spec_passes(float2* z1, float2* z2, const float2* tw, int tid)
{
    if constexpr (S < N) {
        constexpr int R = N / S >= 16 ? 16 : N / S;
        spec_pass<R, false, T, STRIDE>(z1, z2, nullptr, 0, N, S, tw, tid);
        spec_passes<N, S * R, T, STRIDE>(z1, z2, tw, tid);
    }
}

constexpr int spec_threads(int N) { return N / 16 > 128 ? N / 16 : 128; }
// resident CTAs per SM the kernel is compiled for: 512 threads per SM (128 registers a thread)
constexpr int spec_min_blocks(int N) { return 512 / spec_threads(N); }

// One CTA per cell, spec_threads(N) threads.  Shared memory: Z1 and Z2 (N elements each, padded)
// and the N/2 twiddles.  The first pass reads the cell's bins from global memory (consecutive
// threads, consecutive bins); the power of frequency k needs Z1 at k and N - k, so it is formed
// from shared memory after the last pass.  (A CTA looping over cells keeps every pass's state
// live across the loop and spills; a fresh CTA per cell fits the registers, and reloading the
// twiddles from L2 costs N/2 x 8 bytes per cell.)
template <int N, typename T, int STRIDE>
__global__ void __launch_bounds__(spec_threads(N), spec_min_blocks(N)) k_spectrum_fused(const T* __restrict__ fields,
                                                                                        int c0,
                                                                                        const float2* __restrict__ tw_g,
                                                                                        float scale, float* __restrict__ P)
{
    extern __shared__ float2 sm[];
    constexpr int zlen = N + N / 16;
    constexpr int R1 = N >= 16 ? 16 : N;
    float2* z1 = sm;
    float2* z2 = sm + zlen;
    float2* tw = sm + 2 * zlen;
    const int tid = threadIdx.x;
    const size_t cell = blockIdx.x;
    const T* row = fields + cell * N * STRIDE;
    // filled before the first pass's barrier, read after it
    for (int j = tid; j < N / 2; j += blockDim.x) tw[j] = tw_g[j];
    spec_pass<R1, true, T, STRIDE>(z1, z2, row, c0, N, 1, tw, tid);
    spec_passes<N, R1, T, STRIDE>(z1, z2, tw, tid);
    constexpr int nk = N / 2 + 1;
    float* out = P + cell * nk;
    for (int k = tid; k < nk; k += blockDim.x) {
        const int km = (N - k) & (N - 1);
        const float2 a = z1[pad(k)], am = z1[pad(km)], c = z2[pad(k)];
        const float pxy = 0.5f * (a.x * a.x + a.y * a.y + am.x * am.x + am.y * am.y);
        out[k] = scale * (pxy + (c.x * c.x + c.y * c.y));
    }
}

template <int N, typename T, int STRIDE>
cudaError_t launch_fused_n(const T* fields, int n_pix, int c0, const float2* tw, float scale, float* P,
                           cudaStream_t s)
{
    constexpr int threads = spec_threads(N);
    const size_t smem = sizeof(float2) * (2 * (size_t)(N + N / 16) + N / 2);
    auto k = k_spectrum_fused<N, T, STRIDE>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k<<<n_pix, threads, smem, s>>>(fields, c0, tw, scale, P);
    return cudaGetLastError();
}

template <typename T, int STRIDE>
cudaError_t launch_fused(const T* fields, int n_pix, int N, int c0, const float2* tw, float scale, float* P,
                         cudaStream_t s)
{
    switch (N) {
    case 2: return launch_fused_n<2, T, STRIDE>(fields, n_pix, c0, tw, scale, P, s);
    case 4: return launch_fused_n<4, T, STRIDE>(fields, n_pix, c0, tw, scale, P, s);
    case 8: return launch_fused_n<8, T, STRIDE>(fields, n_pix, c0, tw, scale, P, s);
    case 16: return launch_fused_n<16, T, STRIDE>(fields, n_pix, c0, tw, scale, P, s);
    case 32: return launch_fused_n<32, T, STRIDE>(fields, n_pix, c0, tw, scale, P, s);
    case 64: return launch_fused_n<64, T, STRIDE>(fields, n_pix, c0, tw, scale, P, s);
    case 128: return launch_fused_n<128, T, STRIDE>(fields, n_pix, c0, tw, scale, P, s);
    case 256: return launch_fused_n<256, T, STRIDE>(fields, n_pix, c0, tw, scale, P, s);
    case 512: return launch_fused_n<512, T, STRIDE>(fields, n_pix, c0, tw, scale, P, s);
    case 1024: return launch_fused_n<1024, T, STRIDE>(fields, n_pix, c0, tw, scale, P, s);
    case 2048: return launch_fused_n<2048, T, STRIDE>(fields, n_pix, c0, tw, scale, P, s);
    case 4096: return launch_fused_n<4096, T, STRIDE>(fields, n_pix, c0, tw, scale, P, s);
    case 8192: return launch_fused_n<8192, T, STRIDE>(fields, n_pix, c0, tw, scale, P, s);
    default: return cudaErrorInvalidValue;
    }
}

// ---------------------------------------------------------------------------------------------
// Long series: n = n1 N2 + n2, k = k1 + N1 k2,
//   X[k1 + N1 k2] = sum_{n2} w_{N2}^{n2 k2} [ w_N^{n2 k1} sum_{n1} w_{N1}^{n1 k1} x[n1 N2 + n2] ].
// k_split_columns forms the bracket Y[k1][n2] for C = 4096 / N1 neighbouring columns n2 per CTA (each row n1
// of them is C consecutive bins), k_split_rows the sums over n2 for rows k1 and N1 - k1, which hold the
// frequencies k and N - k that the power of Z1 = F_x + i F_y needs together; Z2 = F_z is real, so its rows
// k1 <= N1 / 2 suffice.  Bound by memory: 32 bytes read per bin and cell (whole sectors), 12 written and
// read again for Y, 2 written for the power.  Cells go through both kernels in batches whose Y fits L2, so
// only the bins and the power touch DRAM.  Measured, 512 cells x 131072 bins: 6.12 ms as 17 radix-2 passes
// over the batch (4.3 GB each) plus packing and power; 0.90 ms in two kernels per batch of 42 cells (columns
// 0.52 ms, 4.1 TB/s of the bins; rows 0.38 ms).  The fixed roots of the in-register transforms and the roots
// between the kernels carry FP32's remainders: every butterfly multiplies by the same few roots, so their
// rounding adds up where radix-2 passes average over a table.  Relative L2 error of the power of noise
// against FP64, N = 2^14 / 2^17 / 2^22: radix-2 passes 1.29 / 1.38 / 1.50e-7, here 1.15 / 1.19 / 1.32e-7, and
// 1.66 / 1.82 / 2.12e-7 with roots rounded to FP32, at the same speed (bound by memory).
// ---------------------------------------------------------------------------------------------
constexpr int kColumnElems = 4096;      // elements of each of Z1, Z2 per CTA of k_split_columns, 16 per thread
constexpr int kColumnThreads = kColumnElems / 16;

// a (h + l) for a root h of FP32 digits and its small remainder l: the remainder joins the smaller product
// before its rounding.
__device__ __forceinline__ float2 cmul_comp(float2 a, float2 h, float2 l)
{
    const float x = __fmaf_rn(a.y, h.y, __fmaf_rn(a.y, l.y, -__fmul_rn(a.x, l.x)));
    const float y = __fmaf_rn(a.y, h.x, __fmaf_rn(a.y, l.x, __fmul_rn(a.x, l.y)));
    return make_float2(__fmaf_rn(a.x, h.x, -x), __fmaf_rn(a.x, h.y, y));
}

// h and l with h + l = exp(-2 pi i e / N), e < N: h the table's root exp(-2 pi i j / N1) at the nearest multiple
// j of N / N1 = N2, l = its lo part plus h (exp(-i theta) - 1), |theta| <= pi / N1 < 0.1, by the power series
// (the first terms left out are theta^7 / 5040 < 2e-11 and theta^8 / 40320).  (sincospif's value is off by up
// to an ulp, which the transform's error showed.)
template <int N1>
__device__ __forceinline__ void split_root(const float2* tw, int e, int N2, float two_over_n, float2& h, float2& l)
{
    const int log2_n2 = 31 - __clz(N2), j = (e + N2 / 2) >> log2_n2;
    const float th = 3.14159265358979f * (two_over_n * (float)(e - (j << log2_n2))), t2 = th * th;
    const float sn = th * (1.f - t2 * (1.f / 6.f - t2 * (1.f / 120.f)));
    const float vc = t2 * (0.5f - t2 * (1.f / 24.f - t2 * (1.f / 720.f)));          // 1 - cos
    const bool neg = j & (N1 / 2);
    const int i = j & (N1 / 2 - 1);
    const float2 a = tw[i], b = tw[N1 / 2 + i];
    h = neg ? make_float2(-a.x, -a.y) : a;
    const float2 lo = neg ? make_float2(-b.x, -b.y) : b;
    l = make_float2(lo.x + (h.y * sn - h.x * vc), lo.y - (h.x * sn + h.y * vc));
}

// One Stockham pass (see spec_pass) of radix R at stride S over the columns of both transforms, rows of
// C elements in shared memory (row i at pad(i)); LAST: the results go to global memory, multiplied by
// exp(-2 pi i n2 k1 / N).  tw: exp(-2 pi i j / N1), j < N1 / 2, rounded to FP32, then the remainders.
template <int N1, int S, typename T, int STRIDE>
__device__ __forceinline__ void column_passes(float2* z1, float2* z2, const float2* tw, const T* row, int c0, int N2,
                                              int n2, float two_over_n, float2* Y1, float2* Y2)
{
    constexpr int C = kColumnElems / N1, R = N1 / S >= 16 ? 16 : N1 / S, NB = 16 / R;
    constexpr int n = N1 / S, m = n / R;
    constexpr bool LAST = S * R == N1;
    const int c = threadIdx.x % C, t = threadIdx.x / C;
    float2 a1[NB][R], a2[NB][R];
#pragma unroll
    for (int u = 0; u < NB; ++u) {
        const int b = t + u * (N1 / 16), q = b % S, p = b / S;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int i = q + S * (p + r * m);
            if (S == 1) {
                const float3 v = Load3<T, STRIDE>::get(row, i * N2 + n2, c0);
                a1[u][r] = make_float2(v.x, v.y);
                a2[u][r] = make_float2(v.z, 0.f);
            } else {
                a1[u][r] = z1[pad(i) * C + c];
                a2[u][r] = z2[pad(i) * C + c];
            }
        }
    }
    if (S > 1) __syncthreads();         // every read of the pass is done
#pragma unroll
    for (int u = 0; u < NB; ++u) {
        const int b = t + u * (N1 / 16), q = b % S, p = b / S;
        dft_bitrev<R>(a1[u]);
        dft_bitrev<R>(a2[u]);
        const int o = q + S * R * p;
#pragma unroll
        for (int k = 0; k < R; ++k) {
            float2 b1 = a1[u][bitrev<R>(k)], b2 = a2[u][bitrev<R>(k)];
            const int i = o + S * k;
            if (LAST) {                 // m = 1, p = 0: no twiddle of its own; i = k1
                float2 wh, wl;
                split_root<N1>(tw, i * n2, N2, two_over_n, wh, wl);
                Y1[(size_t)i * N2 + n2] = cmul_comp(b1, wh, wl);
                if (i <= N1 / 2) Y2[(size_t)i * N2 + n2] = cmul_comp(b2, wh, wl);
            } else {
                if (k > 0) {
                    const float2 w = twiddle(tw, p * k * S, N1 / 2);
                    b1 = cmul(b1, w);
                    b2 = cmul(b2, w);
                }
                z1[pad(i) * C + c] = b1;
                z2[pad(i) * C + c] = b2;
            }
        }
    }
    if constexpr (!LAST) {
        __syncthreads();
        column_passes<N1, S * R, T, STRIDE>(z1, z2, tw, row, c0, N2, n2, two_over_n, Y1, Y2);
    }
}

constexpr size_t split_columns_smem(int N1)
{
    return sizeof(float2) * (2 * (size_t)(N1 + N1 / 16) * (kColumnElems / N1) + N1);
}

// grid (N2 / C, cells); tab: exp(-2 pi i j / M), j < M / 2, M = N1 tab_step, rounded to FP32, then the remainders
template <int N1, typename T, int STRIDE>
__global__ void __launch_bounds__(kColumnThreads, 2) k_split_columns(const T* __restrict__ fields, int c0, int N2,
                                                                     const float2* __restrict__ tab, int tab_step,
                                                                     float2* __restrict__ Y1, float2* __restrict__ Y2)
{
    extern __shared__ float2 sm[];
    constexpr int C = kColumnElems / N1, zlen = (N1 + N1 / 16) * C;
    float2* tw = sm + 2 * zlen;
    for (int j = threadIdx.x; j < N1; j += kColumnThreads) tw[j] = tab[j * tab_step];       // (the halves of tab too)
    __syncthreads();
    const size_t cell = blockIdx.y;
    const int n2 = blockIdx.x * C + threadIdx.x % C;
    const size_t N = (size_t)N1 * N2;
    column_passes<N1, 1, T, STRIDE>(sm, sm + zlen, tw, fields + cell * N * STRIDE, c0, N2, n2, 2.f / (float)N,
                                    Y1 + cell * N, Y2 + cell * (size_t)(N1 / 2 + 1) * N2);
}

// Rows: one Stockham pass over the three rows (Z1 at k1 and N1 - k1, Z2 at k1) of a row pair.
template <int N2, int S>
__device__ __forceinline__ void row_passes(float2* const (&z)[3], const float2* const (&src)[3], const float2* tw,
                                           int t)
{
    constexpr int R = N2 / S >= 16 ? 16 : N2 / S, NB = 16 / R, m = N2 / S / R;
    float2 a[3][NB][R];
#pragma unroll
    for (int v = 0; v < 3; ++v)
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            const int b = t + u * (N2 / 16), q = b % S, p = b / S;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int i = q + S * (p + r * m);
                a[v][u][r] = S == 1 ? __ldg(src[v] + i) : z[v][pad(i)];
            }
        }
    __syncthreads();                    // every read of the pass is done (first pass: tw is filled)
#pragma unroll
    for (int u = 0; u < NB; ++u) {
        const int b = t + u * (N2 / 16), q = b % S, p = b / S;
        const int o = q + S * R * p;
#pragma unroll
        for (int v = 0; v < 3; ++v) dft_bitrev<R>(a[v][u]);
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const float2 w = (m > 1 && k > 0) ? twiddle(tw, p * k * S, N2 / 2) : make_float2(1.f, 0.f);
#pragma unroll
            for (int v = 0; v < 3; ++v) {
                const float2 x = a[v][u][bitrev<R>(k)];
                z[v][pad(o + S * k)] = (m > 1 && k > 0) ? cmul(x, w) : x;
            }
        }
    }
    __syncthreads();
    if constexpr (S * R < N2) row_passes<N2, S * R>(z, src, tw, t);
}

constexpr int row_pairs(int N2) { return N2 >= 4096 ? 1 : 4096 / N2; }          // per CTA
constexpr int row_threads(int N2) { return row_pairs(N2) * (N2 / 16); }
// row stride in shared memory: 16 bytes beyond a multiple of 128, so that neighbouring rows' elements at
// one index (the power step) lie on different banks
constexpr int row_stride(int N2) { return N2 + N2 / 16 + 2; }
constexpr size_t split_rows_smem(int N2)
{
    return sizeof(float2) * (3 * (size_t)row_pairs(N2) * row_stride(N2) + N2 / 2);
}

// grid (ceil((N1 / 2 + 1) / row_pairs), cells)
template <int N2>
__global__ void __launch_bounds__(row_threads(N2), N2 <= 2048 ? 2 : 1)
    k_split_rows(const float2* __restrict__ Y1, const float2* __restrict__ Y2, int N1, const float2* __restrict__ tab,
                 int tab_step, float scale, float* __restrict__ P)
{
    extern __shared__ float2 sm[];
    constexpr int G = row_pairs(N2), TT = N2 / 16, LD = row_stride(N2);
    float2* tw = sm + 3 * G * LD;
    for (int j = threadIdx.x; j < N2 / 2; j += row_threads(N2)) tw[j] = tab[j * tab_step];
    const size_t N = (size_t)N1 * N2, cell = blockIdx.y;
    const int first = blockIdx.x * G, half = N1 / 2;
    const int g = threadIdx.x / TT, t = threadIdx.x % TT;
    const int k1 = min(first + g, half);                // (a surplus row pair repeats the last)
    const float2* const src[3] = {Y1 + cell * N + (size_t)k1 * N2, Y1 + cell * N + (size_t)((N1 - k1) % N1) * N2,
                                  Y2 + (cell * (half + 1) + k1) * N2};
    float2* const z[3] = {sm + (3 * g) * LD, sm + (3 * g + 1) * LD, sm + (3 * g + 2) * LD};
    row_passes<N2, 1>(z, src, tw, t);
    float* out = P + cell * (N / 2 + 1);
    for (int e = threadIdx.x; e < G * N2; e += row_threads(N2)) {
        const int h = e % G, k2 = e / G, kk = first + h;
        if (kk > half) continue;
        const float2* zr = sm + 3 * h * LD;
        // N - k: row N1 - k1, element N2 - 1 - k2 (row 0: N2 - k2)
        const int mir = kk == 0 ? (N2 - k2) & (N2 - 1) : N2 - 1 - k2;
        const float2 a = zr[pad(k2)], b = zr[LD + pad(mir)], c = zr[2 * LD + pad(k2)];
        const float pxy = 0.5f * (a.x * a.x + a.y * a.y + b.x * b.x + b.y * b.y);
        const size_t k = (size_t)kk + (size_t)N1 * k2;
        // rows 0 and N1 / 2 hold both k and N - k, whose sums may differ in the last digit: only k <= N / 2
        // writes there, so that every frequency has one writer
        if (k > N / 2 && (kk == 0 || kk == half)) continue;
        out[k <= N / 2 ? k : N - k] = scale * (pxy + (c.x * c.x + c.y * c.y));
    }
}

int split_n2(int N) { return N <= 131072 ? 512 : std::min(4096, N / 256); }

// cells per batch: their Y (12 bytes per bin and cell and a little more) within 64 MB of L2
int split_batch(int n_pix, int N)
{
    const long long per_cell = 12LL * N + 8LL * split_n2(N);
    return (int)std::max(1LL, std::min<long long>(n_pix, (64LL << 20) / per_cell));
}

template <int N1, typename T, int STRIDE>
cudaError_t launch_columns(const T* fields, int cells, int c0, int N2, const float2* tab, int M, float2* Y1, float2* Y2,
                           cudaStream_t s)
{
    auto k = k_split_columns<N1, T, STRIDE>;
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)split_columns_smem(N1));
    if (e != cudaSuccess) return e;
    k<<<dim3(N2 / (kColumnElems / N1), cells), kColumnThreads, split_columns_smem(N1), s>>>(fields, c0, N2, tab, M / N1,
                                                                                           Y1, Y2);
    return cudaGetLastError();
}

template <int N2>
cudaError_t launch_rows(const float2* Y1, const float2* Y2, int cells, int N1, const float2* tab, int M, float scale,
                        float* P, cudaStream_t s)
{
    auto k = k_split_rows<N2>;
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)split_rows_smem(N2));
    if (e != cudaSuccess) return e;
    const int pairs = N1 / 2 + 1, G = row_pairs(N2);
    k<<<dim3((pairs + G - 1) / G, cells), row_threads(N2), split_rows_smem(N2), s>>>(Y1, Y2, N1, tab, M / N2, scale, P);
    return cudaGetLastError();
}

template <typename T, int STRIDE>
cudaError_t launch_split(const T* fields, int n_pix, int N, int c0, float2* work, const float2* tab, float scale, float* P,
                         cudaStream_t s)
{
    const int N2 = split_n2(N), N1 = N / N2, M = std::max(N1, N2), batch = split_batch(n_pix, N);
    float2* Y1 = work;
    float2* Y2 = work + (size_t)batch * N;
    for (int j = 0; j < n_pix; j += batch) {
        const int cells = std::min(batch, n_pix - j);
        const T* f = fields + (size_t)j * N * STRIDE;
        float* out = P + (size_t)j * (N / 2 + 1);
        cudaError_t e = cudaErrorInvalidValue;
        switch (N1) {
        case 32: e = launch_columns<32, T, STRIDE>(f, cells, c0, N2, tab, M, Y1, Y2, s); break;
        case 64: e = launch_columns<64, T, STRIDE>(f, cells, c0, N2, tab, M, Y1, Y2, s); break;
        case 128: e = launch_columns<128, T, STRIDE>(f, cells, c0, N2, tab, M, Y1, Y2, s); break;
        case 256: e = launch_columns<256, T, STRIDE>(f, cells, c0, N2, tab, M, Y1, Y2, s); break;
        case 512: e = launch_columns<512, T, STRIDE>(f, cells, c0, N2, tab, M, Y1, Y2, s); break;
        case 1024: e = launch_columns<1024, T, STRIDE>(f, cells, c0, N2, tab, M, Y1, Y2, s); break;
        default: break;
        }
        if (e != cudaSuccess) return e;
        e = cudaErrorInvalidValue;
        switch (N2) {
        case 512: e = launch_rows<512>(Y1, Y2, cells, N1, tab, M, scale, out, s); break;
        case 1024: e = launch_rows<1024>(Y1, Y2, cells, N1, tab, M, scale, out, s); break;
        case 2048: e = launch_rows<2048>(Y1, Y2, cells, N1, tab, M, scale, out, s); break;
        case 4096: e = launch_rows<4096>(Y1, Y2, cells, N1, tab, M, scale, out, s); break;
        default: break;
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

int grid_for(long long n, int threads) { return grid_stride_blocks(n, threads, 32); }

}  // namespace

void fill_twiddles(float2* host, int M, bool remainders)
{
    const double two_pi = 6.283185307179586476925287;
    for (int j = 0; j < M / 2; ++j) {
        const double a = -two_pi * (double)j / (double)M, c = cos(a), s = sin(a);
        host[j] = make_float2((float)c, (float)s);
        if (remainders) host[M / 2 + j] = make_float2((float)(c - (double)host[j].x), (float)(s - (double)host[j].y));
    }
}

bool spectrum_fused(int N) { return N >= 2 && N <= kFusedMaxN; }
bool spectrum_split(int N) { return N > kFusedMaxN && N <= kSplitMaxN; }

int spectrum_twiddle_length(int N)
{
    return spectrum_split(N) ? std::max(split_n2(N), N / split_n2(N)) : N;
}

size_t spectrum_work_bytes(int n_pix, int N)
{
    if (spectrum_fused(N)) return 0;
    if (spectrum_split(N)) {
        const size_t N2 = split_n2(N), N1 = N / N2;
        return sizeof(float2) * (size_t)split_batch(n_pix, N) * ((size_t)N + (N1 / 2 + 1) * N2);
    }
    return 2 * sizeof(float2) * 2 * (size_t)n_pix * N;
}

// work: spectrum_work_bytes; tw: exp(-2 pi i j / M), j < M / 2, M = spectrum_twiddle_length(N) (split
// transforms: then the M / 2 remainders of rounding them to FP32).
cudaError_t launch_power_spectrum(const void* fields, int precision, int n_pix, int N, int c0, float2* work,
                                  const float2* tw, float scale, float* P, cudaStream_t s)
{
    if (spectrum_split(N)) {
        if (precision == RD_MIXED)
            return launch_split<float, 8>(static_cast<const float*>(fields), n_pix, N, c0, work, tw, scale, P, s);
        return launch_split<double, 6>(static_cast<const double*>(fields), n_pix, N, c0, work, tw, scale, P, s);
    }
    if (spectrum_fused(N)) {
        if (precision == RD_MIXED)
            return launch_fused<float, 8>(static_cast<const float*>(fields), n_pix, N, c0, tw, scale, P, s);
        return launch_fused<double, 6>(static_cast<const double*>(fields), n_pix, N, c0, tw, scale, P, s);
    }
    static_assert(kMixedMaxBins <= kSplitMaxN, "series of RD_MIXED detectors take one of the above");
    if (precision == RD_MIXED) return cudaErrorInvalidValue;
    float2* z = work;                                   // two arrays [2 n_pix][N]
    float2* y = work + 2 * (size_t)n_pix * N;
    k_pack_spectrum_input<<<grid_for((long long)n_pix * N, 256), 256, 0, s>>>(static_cast<const double*>(fields), n_pix, N,
                                                                             c0, z);
    cudaError_t e = cudaGetLastError();
    float2* a = z;
    float2* b = y;
    const long long batch = 2LL * n_pix;
    for (int st = 1; st < N && e == cudaSuccess; st <<= 1) {
        k_fft_pass<<<grid_for(batch * (N / 2), 256), 256, 0, s>>>(a, b, N, st, tw, batch);
        e = cudaGetLastError();
        float2* t = a;
        a = b;
        b = t;
    }
    if (e != cudaSuccess) return e;
    const long long np = (long long)n_pix * (N / 2 + 1);
    k_spectrum_power<<<grid_for(np, 256), 256, 0, s>>>(a, n_pix, N, scale, P);
    return cudaGetLastError();
}

}  // namespace rd
