// Run-time coupling (Section 3.1: the deposit as a sub-step right after the particle push): a
// Boris pusher for charges in a uniform magnetic field, advancing the state on the device and
// writing the new samples where rd_deposit_stream takes them.
//
// Per step (c = 1, u = gamma beta, magnetic field only, so gamma is constant):
//   t = (qm dt / 2) B / gamma,  s = 2 t / (1 + |t|^2),  u' = u + u x t,  u <- u + u' x s,
//   x <- x + dt u / gamma
// (the Boris rotation: |u| is kept, and u turns about B by 2 atan(|t|) per step).
#include <math.h>

#include "rd_internal.cuh"

namespace rd {

namespace {

__global__ void k_push_boris(int n_part, int n_steps, double dt, double bx, double by, double bz, double qm,
                             double* __restrict__ x, double* __restrict__ u, double* __restrict__ x_out,
                             double* __restrict__ u_out)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n_part) return;
    double X[3] = {x[3 * p], x[3 * p + 1], x[3 * p + 2]};
    double U[3] = {u[3 * p], u[3 * p + 1], u[3 * p + 2]};
    const double g = sqrt(1.0 + (U[0] * U[0] + U[1] * U[1] + U[2] * U[2]));
    const double h = 0.5 * qm * dt / g;
    const double t[3] = {h * bx, h * by, h * bz};
    const double f = 2.0 / (1.0 + (t[0] * t[0] + t[1] * t[1] + t[2] * t[2]));
    const double s[3] = {f * t[0], f * t[1], f * t[2]};
    const double w = dt / g;
    for (int k = 0; k < n_steps; ++k) {
        const double v[3] = {U[0] + (U[1] * t[2] - U[2] * t[1]), U[1] + (U[2] * t[0] - U[0] * t[2]),
                             U[2] + (U[0] * t[1] - U[1] * t[0])};
        U[0] += v[1] * s[2] - v[2] * s[1];
        U[1] += v[2] * s[0] - v[0] * s[2];
        U[2] += v[0] * s[1] - v[1] * s[0];
        X[0] += w * U[0];
        X[1] += w * U[1];
        X[2] += w * U[2];
        const size_t o = ((size_t)p * n_steps + k) * 3;
        x_out[o] = X[0];
        x_out[o + 1] = X[1];
        x_out[o + 2] = X[2];
        u_out[o] = U[0];
        u_out[o + 1] = U[1];
        u_out[o + 2] = U[2];
    }
    x[3 * p] = X[0];
    x[3 * p + 1] = X[1];
    x[3 * p + 2] = X[2];
    u[3 * p] = U[0];
    u[3 * p + 1] = U[1];
    u[3 * p + 2] = U[2];
}

// One thread per value (particle, staged sample, component) of x and u.  A streamed call is a few
// microseconds of copying: one launch instead of seven strided copies (256 particles x 25 samples: 12 us and
// seven enqueues a call, 3 us and one).
__global__ void k_stream_gather(long long total, long long m3, int have3, int kept3, const double* __restrict__ lx,
                                const double* __restrict__ lu, const double* __restrict__ x,
                                const double* __restrict__ u, double* xs, double* us, double* __restrict__ nx,
                                double* __restrict__ nu)
{
    // a particle's staged values: 64 bits hold them for any int32 number of samples (the 64-bit division is ten
    // times longer, so it is left to the calls that need it)
    const long long row = m3 + have3;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const long long p = total <= 0x7fffffffLL ? (int)e / (int)row : e / row;
        const long long r = e - p * row;
        double vx, vu;
        if (r < have3) {
            vx = lx[p * have3 + r];
            vu = lu[p * have3 + r];
        } else if (x) {
            vx = x[p * m3 + (r - have3)];
            vu = u[p * m3 + (r - have3)];
        } else {
            vx = xs[e];
            vu = us[e];
        }
        if (r < have3 || x) {
            xs[e] = vx;
            us[e] = vu;
        }
        if (r >= row - kept3) {
            nx[p * kept3 + (r - (row - kept3))] = vx;
            nu[p * kept3 + (r - (row - kept3))] = vu;
        }
    }
}

}  // namespace

cudaError_t launch_stream_gather(int n_part, int m, int have, int kept, const double* lx, const double* lu,
                                 const double* x, const double* u, double* xs, double* us, double* nx, double* nu,
                                 cudaStream_t s)
{
    const long long total = 3LL * n_part * ((long long)m + have);
    k_stream_gather<<<grid_stride_blocks(total, 256, 8), 256, 0, s>>>(total, 3LL * m, 3 * have, 3 * kept, lx, lu, x, u, xs,
                                                                      us, nx, nu);
    return cudaGetLastError();
}

cudaError_t launch_push_boris(int n_part, int n_steps, double dt, const double* B, double qm, double* x, double* u,
                              double* x_out, double* u_out, cudaStream_t s)
{
    if (n_part <= 0 || n_steps <= 0) return cudaSuccess;
    // one-warp CTAs while they do not fill the multiprocessors: the warps of a CTA share one SM's FP64 pipe
    // (256 particles x 25 steps: 24 us in two CTAs of 128 threads, 9 us in eight of 32)
    const int threads = n_part <= 4 * 32 * sm_count() ? 32 : 128;
    k_push_boris<<<(n_part + threads - 1) / threads, threads, 0, s>>>(n_part, n_steps, dt, B[0], B[1], B[2], qm, x, u,
                                                                      x_out, u_out);
    return cudaGetLastError();
}

}  // namespace rd
