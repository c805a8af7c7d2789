// Per-sample precompute (both precisions), the plain FP64 deposit and the field readout and
// write-in (the mixed-precision deposit is in rd_mixed.cu).
//
// Work decomposition of the FP64 deposit: one CTA = 256 detector cells (one per thread) x one
// particle x one chunk of consecutive intervals.  The chunk's per-sample records are streamed
// through shared memory in tiles of 64 samples by bulk asynchronous copies (double buffered,
// mbarrier completion); every thread reads each record as a broadcast.  Each thread evaluates its
// cell's arrival time from Eq. 2 for every sample (they increase for sub-luminal chords), keeps
// the bin it is filling in registers and adds the bin to global memory only when its arrival time
// leaves the bin.  The FP64 pipe is the bound (on GB300 it runs at 1.6 % of the FP32 rate), so in a
// warp whose lanes all walk a cell, the FP64 work of the few lanes that start a new bin is spread
// over the warp by shuffles and the bin-edge tests run on the integer pipe (fp64_deposit_warp).
#include <math.h>

#include "rd_internal.cuh"

namespace rd {

// =============================================================================================
// Algorithm 1, per-sample part: beta, betadot (backward difference), 1/gamma^2, chord velocity.
// =============================================================================================
__device__ __forceinline__ void beta_of(const double* u, double& bx, double& by, double& bz,
                                        double& ig2)
{
    const double ux = u[0], uy = u[1], uz = u[2];
    const double uu = ux * ux + uy * uy + uz * uz;
    const double g = sqrt(1.0 + uu);
    bx = ux / g;
    by = uy / g;
    bz = uz / g;
    ig2 = 1.0 / (1.0 + uu);
}

// The precompute kernels take one sample per lane; a warp covers 31 samples and its lane 0 the one
// before them, so that the previous sample's beta comes from the neighbouring lane by a shuffle instead
// of a second evaluation (square root and divisions in FP64, the pipe that bounds these kernels: 4e6
// samples took 1274 us, five times the time of their bytes).  Returns the flat sample index (particle *
// n_samples + k) of the lane, -1 beyond the ends; `out` says whether the lane owns the sample.
__device__ __forceinline__ long long warp_sample(long long total, bool& out)
{
    const long long w = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const long long i = w * kPrecomputeSpan - 1 + lane;
    out = lane > 0 && i < total;
    return i < total ? i : -1;
}

// particle and sample of a flat index (32-bit division where it fits: the 64-bit one is ten times longer)
__device__ __forceinline__ void split_sample(long long i, int n_samples, long long& p, int& k)
{
    if (i <= 0xffffffffLL) {
        const unsigned q = (unsigned)i / (unsigned)n_samples;
        p = q;
        k = (int)((unsigned)i - q * (unsigned)n_samples);
    } else {
        p = i / n_samples;
        k = (int)(i - p * n_samples);
    }
}

// not finite (infinity or NaN), tested on the exponent bits (integer pipe)
__device__ __forceinline__ bool not_finite(double v) { return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000; }

__device__ __forceinline__ bool bad3(const double* v) { return not_finite(v[0]) || not_finite(v[1]) || not_finite(v[2]); }

__global__ void k_precompute_mixed(const double* __restrict__ x, const double* __restrict__ u,
                                   const double* __restrict__ q, double qscale, long long total, int n_samples,
                                   double dt, int flags, RecS* __restrict__ rec, DevCounters* counters)
{
    const bool near_on = (flags & RD_NEAR) != 0, far_on = (flags & RD_FAR) != 0;
    const double inv_dt = 1.0 / dt;
    bool out;
    const long long i = warp_sample(total, out);
    double xk[3] = {0.0, 0.0, 0.0}, uk[3] = {0.0, 0.0, 0.0};
    if (i >= 0) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            xk[c] = x[3 * i + c];
            uk[c] = u[3 * i + c];
        }
    }
    // beta = u / gamma, gamma^-1 = (1 + u^2)^(-1/2): the records are FP32, one ulp of FP64 more or less
    // in gamma^-1 does not show in them
    const double rg = rsqrt(fma(uk[0], uk[0], fma(uk[1], uk[1], fma(uk[2], uk[2], 1.0))));
    const double ig2 = rg * rg;
    double b[3], db[3], dx[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        b[c] = uk[c] * rg;
        db[c] = b[c] - __shfl_up_sync(0xffffffffu, b[c], 1);
        dx[c] = xk[c] - __shfl_up_sync(0xffffffffu, xk[c], 1);
    }
    if (!out) return;
    long long p;
    int k;
    split_sample(i, n_samples, p, k);
    // charge factor folded into the betadot and gamma^-2 terms of Eq. 1 (deposit records)
    const double qf = qscale != 0.0 ? -(q ? q[p] : 1.0) * qscale : 1.0;
    bool bad = bad3(xk) || bad3(uk);
    double v[3] = {0.0, 0.0, 0.0}, g = 1.0;
    if (k == 0) {
        db[0] = db[1] = db[2] = 0.0;
    } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) v[c] = dx[c] * inv_dt;
        g = fma(-v[0], v[0], fma(-v[1], v[1], fma(-v[2], v[2], 1.0)));
        bad = bad || !(g > 0.0);
    }
    if (bad) atomicOr(&counters->errors, ERRBIT_INPUT);
    // e = beta_k - vbar_k (difference of end-point and chord velocities)
    const double e[3] = {b[0] - v[0], b[1] - v[1], b[2] - v[2]};
    const double qa = far_on ? qf * inv_dt : 0.0;
    RecS r;
    r.nx = (float)-xk[0];
    r.ny = (float)-xk[1];
    r.nz = (float)-xk[2];
    const float ig2f = (float)ig2;
    r.nhig2 = -0.5f * ig2f;
    r.nbx = (float)-b[0];
    r.nby = (float)-b[1];
    r.nbz = (float)-b[2];
    r.ig2n = near_on ? (float)(qf * ig2) : 0.f;
    r.bdx = (float)(qa * db[0]);
    r.bdy = (float)(qa * db[1]);
    r.bdz = (float)(qa * db[2]);
    r.dtg = (float)(dt * g);
    r.d2x = 2.f * (float)e[0];
    r.d2y = 2.f * (float)e[1];
    r.d2z = 2.f * (float)e[2];
    r.gd = (float)(g + fma(e[0], e[0], fma(e[1], e[1], e[2] * e[2])));
    float4* o = reinterpret_cast<float4*>(rec + i);
    o[0] = make_float4(r.nx, r.ny, r.nz, r.nhig2);
    o[1] = make_float4(r.nbx, r.nby, r.nbz, r.ig2n);
    o[2] = make_float4(r.bdx, r.bdy, r.bdz, r.dtg);
    o[3] = make_float4(r.d2x, r.d2y, r.d2z, r.gd);
}

__global__ void k_precompute_fp64(const double* __restrict__ x, const double* __restrict__ u,
                                  const double* __restrict__ q, long long total, int n_samples, double t0,
                                  double dt, int flags, RecD* __restrict__ rec, DevCounters* counters)
{
    const double near = (flags & RD_NEAR) ? 1.0 : 0.0, far = (flags & RD_FAR) ? 1.0 : 0.0;
    bool out;
    const long long i = warp_sample(total, out);
    double xk[3] = {0.0, 0.0, 0.0}, uk[3] = {0.0, 0.0, 0.0};
    if (i >= 0) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            xk[c] = x[3 * i + c];
            uk[c] = u[3 * i + c];
        }
    }
    double bx, by, bz, ig2;
    beta_of(uk, bx, by, bz, ig2);
    const double px = __shfl_up_sync(0xffffffffu, bx, 1), py = __shfl_up_sync(0xffffffffu, by, 1),
                 pz = __shfl_up_sync(0xffffffffu, bz, 1);
    const double xp[3] = {__shfl_up_sync(0xffffffffu, xk[0], 1), __shfl_up_sync(0xffffffffu, xk[1], 1),
                          __shfl_up_sync(0xffffffffu, xk[2], 1)};
    if (!out) return;
    long long p;
    int k;
    split_sample(i, n_samples, p, k);
    bool bad = bad3(xk) || bad3(uk);
    double ax = 0.0, ay = 0.0, az = 0.0;
    if (k > 0) {
        ax = (bx - px) / dt;
        ay = (by - py) / dt;
        az = (bz - pz) / dt;
        const double vx = xk[0] - xp[0], vy = xk[1] - xp[1], vz = xk[2] - xp[2];
        bad = bad || !((vx * vx + vy * vy) + vz * vz < dt * dt);
    }
    if (bad) atomicOr(&counters->errors, ERRBIT_INPUT);
    RecD r;
    const double qp = q ? q[p] : 1.0;
    r.xa = D4{xk[0], xk[1], xk[2], __dadd_rn(t0, __dmul_rn((double)k, dt))};
    r.bb = D4{bx, by, bz, (near * qp) * ig2};
    r.bd = D4{(far * qp) * ax, (far * qp) * ay, (far * qp) * az, 0.0};
    rec[i] = r;
}

// =============================================================================================
// Plain FP64 deposit: Eq. 1 as printed, Eq. 2 evaluated directly for every sample.
// =============================================================================================
struct D64State {
    int b;
    double a;       // arrival (bins) of the previous sample
    double acc[6];
    double Fp[6];   // RD_LINEAR / RD_QUADRATIC: field of the previous sample
    double Fpp[6];  // RD_QUADRATIC: field two samples back ...
    double ap;      // ... and its arrival (bins)
    double e;       // held field: upper edge of bin b (b + 1) ...
    long long ke;   // ... and its order key (dkey)
    int n_below;
    int n_above;
};

// An integer that orders like the double x (finite x): the bit pattern for x >= 0, the magnitude bits
// flipped for x < 0, so that bin-edge tests run on the integer pipe.
__device__ __forceinline__ long long dkey(double x)
{
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}

__device__ __forceinline__ void set_edge(D64State& st, double e)
{
    st.e = e;
    st.ke = dkey(e);
}

// The double n (|n| < 2^31) assembled from its integer on the integer pipe: sign, exponent
// 1023 + floor(log2 |n|), and the bits of |n| below its leading one as the mantissa's top bits.
__device__ __forceinline__ double int_to_double_bits(int n)
{
    const unsigned m = (unsigned)(n < 0 ? -n : n);
    const int hb = 31 - __clz((int)m);
    const long long bits = ((long long)(n < 0) << 63) | ((long long)(1023 + hb) << 52) |
                           ((long long)(m ^ (1u << hb)) << (52 - hb));
    return __longlong_as_double(n == 0 ? 0LL : bits);
}


__device__ __forceinline__ void flush_f64(double* row, int n_bins, int b, const double* v)
{
    if ((unsigned)b < (unsigned)n_bins) {
        double* p = row + (size_t)b * 6;
#pragma unroll
        for (int i = 0; i < 6; ++i) red_add_f64(p + i, v[i]);
    }
}

// Square root and reciprocal start from the FP32 approximations (relative error below 2^-22): the FP64
// operand's leading bits become a float, and the float result a double, on the integer pipe, which this
// kernel leaves idle, so that FP64 refinement takes 6 and 3 operations (9 and 4 from the FP64
// approximations, good to ~2^-20).  The deposit is bound by the FP64 pipe at 61 operations per (cell,
// interval): with 56, 24 particles x 1200 intervals x 4096 cells take 12.48 ms instead of 13.41.  Operands
// outside FP32's range take the plain forms.
__device__ __forceinline__ bool fp32_range(double v)
{
    // positive, exponent within +-100
    return (unsigned)(__double2hiint(v) - ((1023 - 100) << 20)) < (unsigned)(200 << 20);
}

__device__ __forceinline__ float leading_float(double v)    // v truncated to 24 bits
{
    return __int_as_float(((__double2hiint(v) - (896 << 20)) << 3) | (int)((unsigned)__double2loint(v) >> 29));
}

__device__ __forceinline__ double float_bits_to_double(float v)     // exact, v positive and normal
{
    const int b = __float_as_int(v);
    return __hiloint2double((b >> 3) + (896 << 20), b << 29);
}

// The rare operands' square root.  (The volatile statement keeps the compiler from computing it for every operand and
// selecting: 24 particles x 1200 intervals x 4096 cells 14.23 ms.)
__device__ __forceinline__ double sqrt_plain(double a)
{
    asm volatile("" : "+d"(a));
    return __dsqrt_rn(a);
}

// sqrt(a) rounded to nearest, by Markstein's sequence ("IA-64 and Elementary Functions", 2000): one coupled
// Newton-Raphson step for g -> sqrt(a), h -> 1 / (2 sqrt(a)) takes the error to ~2^-44, and adding the residual
// d = a - g^2 (exact but for its own rounding) times h leaves g + d h within ~2^-86 of sqrt(a), 2^-33 ulp, before the
// last rounding.  Closer than that to a rounding boundary (1 operand in 10^10) the result might be the neighbour, so
// the distance is checked, on the FP32 and integer pipes: d h in ulps of g, less the n whole ulps that the sum moved, is
// what the rounding dropped.  FP32 gives it to (|n| + 1) 2^-22, |n| below 1500; within twice that of half an ulp
// (2 operands in 10^4) the plain form is taken.  12.53 ms in the case above without the check, 12.51 with it.
__device__ __forceinline__ double sqrt_markstein(double a)
{
    if (!fp32_range(a)) return sqrt_plain(a);
    const double y = float_bits_to_double(fast_rsqrt(leading_float(a)));
    double h = __hiloint2double(__double2hiint(y) - (1 << 20), __double2loint(y));      // y / 2
    double g = __dmul_rn(a, y);
    const double r = __fma_rn(-h, g, 0.5);
    g = __fma_rn(g, r, g);
    h = __fma_rn(h, r, h);
    const double d = __fma_rn(-g, g, a);
    const double s = __fma_rn(d, h, g);
    // g in [2^e, 2^(e + 1)); d h / ulp(g) = (d / 4^e) (h 2^(e + 52)), d / 4^e a multiple of 2^-104 below 2^-40 (d = 0 may
    // take either way: s is then the root)
    const int gh = __double2hiint(g), sh = __double2hiint(s), dh = __double2hiint(d);
    const int e20 = (gh & 0x7ff00000) - (1023 << 20);
    const float df = __int_as_float((dh & 0x80000000) | ((((dh & 0x7fffffff) - 2 * e20 - (896 << 20)) << 3) |
                                                         (int)((unsigned)__double2loint(d) >> 29)));
    const float hf = __int_as_float(((__double2hiint(h) + e20 + (52 - 896) * (1 << 20)) << 3) |
                                    (int)((unsigned)__double2loint(h) >> 29));
    const float n = (float)(int)((unsigned)__double2loint(s) - (unsigned)__double2loint(g));
    const float dropped = fabsf(__fmaf_rn(df, hf, -n));
    const bool sure = dropped < __fmaf_rn(fabsf(n) + 1.f, -0x1p-21f, 0.5f) && ((gh ^ sh) & 0x7ff00000) == 0;
    if (!sure) return sqrt_plain(a);
    return s;
}

// 1/d: one third-order step y (1 + e + e^2), e = 1 - d y, takes the approximation (2^-22) to FP64 rounding.
// For the positive, normal arguments the field passes (kappa R >= R / (2 gamma^2)).
__device__ __forceinline__ double rcp_cubic(double d)
{
    double y;
    if (fp32_range(d)) {
        y = float_bits_to_double(fast_rcp(leading_float(d)));
    } else {
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
    }
    double e = fma(-d, y, 1.0);
    e = fma(e, e, e);
    return fma(y, e, y);
}

// Eq. 1 at one cell, with d = x_cell - x_k and R = |d| as computed for the arrival time (Eq. 2).
// Writing n = d / R and kappa R = R - beta.d, Eq. 1 multiplies out to
//   E = q / (kappa R)^3 [a d - R v],   B = n x E = q / (kappa R)^3 v x d,
//   a = gamma^-2 + d.betadot,   v = a beta + (kappa R) betadot,
// so the only reciprocal is 1/(kappa R).  The record holds q gamma^-2 and q betadot, with gamma^-2 = 0
// without the velocity term (RD_NEAR) and betadot = 0 without the acceleration term (RD_FAR), so that
// a and v carry the charge.
__device__ __forceinline__ void fp64_field(const RecD& r, double dx, double dy, double dz, double R, double* F)
{
    const double kR = fma(-r.bb.z, dz, fma(-r.bb.y, dy, fma(-r.bb.x, dx, R)));
    const double a = fma(r.bd.z, dz, fma(r.bd.y, dy, fma(r.bd.x, dx, r.bb.w)));
    const double w = rcp_cubic(kR);
    const double Qk = w * w;                            // q-free (kappa R)^-3 times kappa R
    const double Qa = (w * Qk) * a;
    const double vx = fma(Qa, r.bb.x, Qk * r.bd.x);     // Q v
    const double vy = fma(Qa, r.bb.y, Qk * r.bd.y);
    const double vz = fma(Qa, r.bb.z, Qk * r.bd.z);
    F[0] = fma(Qa, dx, -R * vx);
    F[1] = fma(Qa, dy, -R * vy);
    F[2] = fma(Qa, dz, -R * vz);
    F[3] = fma(vy, dz, -vz * dy);
    F[4] = fma(vz, dx, -vx * dz);
    F[5] = fma(vx, dy, -vy * dx);
}

// Eq. 2 for a record: the cell offset d, R = |d| and the arrival time in bins, with the same
// separately rounded operations as arrival_bins (t_k from the record).
__device__ __forceinline__ double fp64_arrival(const RecD& r, const D4& cl, double inv_dt_det, double& dx,
                                               double& dy, double& dz, double& R)
{
    dx = __dsub_rn(cl.x, r.xa.x);
    dy = __dsub_rn(cl.y, r.xa.y);
    dz = __dsub_rn(cl.z, r.xa.z);
    R = sqrt_markstein(__dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz)));
    return __dmul_rn(__dsub_rn(__dadd_rn(r.xa.w, R), cl.w), inv_dt_det);
}

// Far-field limit of the radiation term: E = q n_c x ((n_c - beta) x betadot) / (kappa^3 R_c),
// kappa = 1 - beta.n_c, B = n_c x E (the record's betadot carries q, and is zero without RD_FAR).
__device__ __forceinline__ void fp64_field_ff(const RecD& r, double nx, double ny, double nz, double Rc,
                                              double* F)
{
    const double mx = nx - r.bb.x, my = ny - r.bb.y, mz = nz - r.bb.z;
    const double kap = 1.0 - (r.bb.x * nx + r.bb.y * ny + r.bb.z * nz);
    const double s = 1.0 / (kap * kap * kap * Rc);
    const double wx = my * r.bd.z - mz * r.bd.y;
    const double wy = mz * r.bd.x - mx * r.bd.z;
    const double wz = mx * r.bd.y - my * r.bd.x;
    const double Ex = s * (ny * wz - nz * wy), Ey = s * (nz * wx - nx * wz), Ez = s * (nx * wy - ny * wx);
    F[0] = Ex;
    F[1] = Ey;
    F[2] = Ez;
    F[3] = ny * Ez - nz * Ey;
    F[4] = nz * Ex - nx * Ez;
    F[5] = nx * Ey - ny * Ex;
}

// Deposit [st.a, c] with the bin-overlap arithmetic of the integrator detector.  The part inside the
// filling bin (up to its upper edge st.e = st.b + 1) is added on every step; only an interval that
// passes the edge flushes the bin and starts the next one with the rest, so the operations that
// every lane of a warp runs stay few (nearly every warp has a lane that crosses on each step).
__device__ __forceinline__ void fp64_deposit(D64State& st, const double* F, double c, double* row,
                                             int n_bins, int k, int k_begin, int k_end)
{
    const bool cr = c >= st.e;
    const double wi = (cr ? st.e : c) - st.a;
#pragma unroll
    for (int i = 0; i < 6; ++i) st.acc[i] = fma(F[i], wi, st.acc[i]);
    if (cr) {
        flush_f64(row, n_bins, st.b, st.acc);
        int b = st.b + 1;
        double e = st.e;                       // lower edge of bin b
        if (c >= e + 1.0) {                    // more than one edge: whole bins in between
            const int bc = clamp_bin(floor(c));
            const int lo = max(b, 0), hi = min(bc - 1, n_bins - 1);
            for (int j = lo; j <= hi; ++j) flush_f64(row, n_bins, j, F);
            b = bc;
            e = (double)bc;
        }
        const double wl = c - e;
#pragma unroll
        for (int i = 0; i < 6; ++i) st.acc[i] = F[i] * wl;
        if (st.b < 0 && b >= 0) st.n_below = k - k_begin + 1;
        if (st.b < n_bins && b >= n_bins) st.n_above = k_end - k + 1;
        st.b = b;
        set_edge(st, e + 1.0);
    }
    st.a = c;
}

// fp64_deposit for a warp whose 32 lanes all walk a cell (`warp` converged on every call).  The
// lanes whose arrival passed their bin's upper edge (about one in five) start their next bin with
// the rest of the interval, F times (c - e): instead of each lane's six multiplies taking six
// warp-wide FP64 instructions, the warp's crossing lanes' products are spread over all 32 lanes by
// shuffles (one or two FP64 instructions); the edge tests are integer compares and the next edge is
// assembled on the integer pipe, so that the FP64 pipe does the arithmetic of Eq. 1 and 2.
__device__ __forceinline__ void fp64_deposit_warp(D64State& st, const double* F, double c, double* row,
                                                  int n_bins, int k, int k_begin, int k_end)
{
    constexpr unsigned warp = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const long long kc = dkey(c);
    const bool cr = kc >= st.ke;
    const double wi = (cr ? st.e : c) - st.a;
#pragma unroll
    for (int i = 0; i < 6; ++i) st.acc[i] = fma(F[i], wi, st.acc[i]);
    st.a = c;
    const unsigned m = __ballot_sync(warp, cr);
    if (m == 0u) return;
    double wl = 0.0;
    if (cr) {
        flush_f64(row, n_bins, st.b, st.acc);
        int b = st.b + 1;
        wl = c - st.e;                         // st.e: lower edge of bin b
        // c - e >= 1 (compared on the bits: both are >= 0): more than one edge, whole bins in between
        if (__double_as_longlong(wl) >= 0x3FF0000000000000LL) {
            const int bc = clamp_bin(floor(c));
            const int lo = max(b, 0), hi = min(bc - 1, n_bins - 1);
            for (int j = lo; j <= hi; ++j) flush_f64(row, n_bins, j, F);
            b = bc;
            wl = c - (double)bc;
        }
        if (st.b < 0 && b >= 0) st.n_below = k - k_begin + 1;
        if (st.b < n_bins && b >= n_bins) st.n_above = k_end - k + 1;
        st.b = b;
        set_edge(st, int_to_double_bits(b + 1));
    }
    // product p = 6 r + q (r: rank of a crossing lane, q: component) is formed by lane p % 32 in
    // round p / 32 and handed back to its crossing lane
    const int n = __popc(m);
    const int rank = __popc(m & ((1u << lane) - 1u));
    for (int base = 0; base < 6 * n; base += 32) {
        const int pi = base + lane;
        const int r = pi / 6, q = pi - 6 * (pi / 6);
        const int src = pi < 6 * n ? (int)__fns(m, 0u, r + 1) : lane;
        double f = 0.0;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            const double v = __shfl_sync(warp, F[i], src);
            f = (q == i) ? v : f;
        }
        const double prod = f * __shfl_sync(warp, wl, src);
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            const int idx = 6 * rank + i;
            const double v = __shfl_sync(warp, prod, idx & 31);
            if (cr && idx >= base && idx < base + 32) st.acc[i] = v;
        }
    }
}

// RD_LINEAR: the field goes linearly from F0 at st.a to F1 at c; the overlap [u0, u1] of the interval
// with a bin weighs F0 (u1 - u0) + (F1 - F0) ((u1 - a)^2 - (u0 - a)^2) / (2 (c - a)).
__device__ __forceinline__ void fp64_lin_part(const double* F0, const double* F1, double a, double c, double u0,
                                              double u1, double* out, bool add)
{
    const double len = u1 - u0;
    const double ramp = ((u1 - a) * (u1 - a) - (u0 - a) * (u0 - a)) / (2.0 * (c - a));
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const double v = F0[i] * len + (F1[i] - F0[i]) * ramp;
        out[i] = add ? out[i] + v : v;
    }
}

__device__ __forceinline__ void fp64_deposit_lin(D64State& st, const double* F0, const double* F1, double c,
                                                 double* row, int n_bins, int k, int k_begin, int k_end)
{
    const double a = st.a;
    const double fc = floor(c);
    const int bc = clamp_bin(fc);
    if (!(c > a)) {
        st.a = c;
        return;
    }
    if (bc <= st.b) {
        fp64_lin_part(F0, F1, a, c, a, c, st.acc, true);
        st.a = c;
        return;
    }
    fp64_lin_part(F0, F1, a, c, a, (double)(st.b + 1), st.acc, true);
    flush_f64(row, n_bins, st.b, st.acc);
    const int lo = max(st.b + 1, 0), hi = min(bc - 1, n_bins - 1);
    for (int j = lo; j <= hi; ++j) {
        double v[6];
        fp64_lin_part(F0, F1, a, c, (double)j, (double)(j + 1), v, false);
        flush_f64(row, n_bins, j, v);
    }
    fp64_lin_part(F0, F1, a, c, fc, c, st.acc, false);
    if (st.b < 0 && bc >= 0) st.n_below = k - k_begin + 1;
    if (st.b < n_bins && bc >= n_bins) st.n_above = k_end - k + 1;
    st.b = bc;
    st.a = c;
}

// RD_QUADRATIC: over [a, c] the quadratic through (p, Fpp), (a, Fa), (c, Fc) in arrival time, in Newton
// form about a (s = tau - a, L = c - a, h = a - p): F(s) = Fa + D1 s + D2 s (s - L), D1 = (Fc - Fa) / L,
// D2 = (D1 - (Fa - Fpp) / h) / (L + h); the overlap [u0, u1] receives
// Fa (s1 - s0) + D1 (s1^2 - s0^2) / 2 + D2 ((s1^3 - s0^3) / 3 - L (s1^2 - s0^2) / 2).
__device__ __forceinline__ void fp64_quad_part(const double* Fa, const double* D1, const double* D2, double a,
                                               double L, double u0, double u1, double* out, bool add)
{
    const double s0 = u0 - a, s1 = u1 - a;
    const double sq = (s1 * s1 - s0 * s0) / 2.0;
    const double cu = (s1 * s1 * s1 - s0 * s0 * s0) / 3.0 - L * sq;
    const double len = u1 - u0;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const double v = Fa[i] * len + D1[i] * sq + D2[i] * cu;
        out[i] = add ? out[i] + v : v;
    }
}

__device__ __forceinline__ void fp64_deposit_quad(D64State& st, const double* Fc, double c, double* row, int n_bins,
                                                  int k, int k_begin, int k_end)
{
    const double a = st.a;
    const double fc = floor(c);
    const int bc = clamp_bin(fc);
    if (!(c > a)) {
        st.a = c;
        return;
    }
    const double L = c - a, h = a - st.ap;
    double D1[6], D2[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const double D0 = (st.Fp[i] - st.Fpp[i]) / h;
        D1[i] = (Fc[i] - st.Fp[i]) / L;
        D2[i] = (D1[i] - D0) / (L + h);
    }
    if (bc <= st.b) {
        fp64_quad_part(st.Fp, D1, D2, a, L, a, c, st.acc, true);
        st.a = c;
        return;
    }
    fp64_quad_part(st.Fp, D1, D2, a, L, a, (double)(st.b + 1), st.acc, true);
    flush_f64(row, n_bins, st.b, st.acc);
    const int lo = max(st.b + 1, 0), hi = min(bc - 1, n_bins - 1);
    for (int j = lo; j <= hi; ++j) {
        double v[6];
        fp64_quad_part(st.Fp, D1, D2, a, L, (double)j, (double)(j + 1), v, false);
        flush_f64(row, n_bins, j, v);
    }
    fp64_quad_part(st.Fp, D1, D2, a, L, fc, c, st.acc, false);
    if (st.b < 0 && bc >= 0) st.n_below = k - k_begin + 1;
    if (st.b < n_bins && bc >= n_bins) st.n_above = k_end - k + 1;
    st.b = bc;
    st.a = c;
}

#ifndef RD_FP64_MINBLOCKS
#define RD_FP64_MINBLOCKS 2      // CTAs of 256 threads per SM the held-field FP64 kernel is compiled for
#endif

// LM: interpolation family, 0 held field (default), 1 linear or held-previous (P.lin 1, 2), 2 quadratic
template <int LM>
__global__ void __launch_bounds__(kDepositThreads, LM == 0 ? RD_FP64_MINBLOCKS : 2) k_deposit_fp64(const DepositParams P,
                                                                       int flags)
{
    __shared__ __align__(128) RecD tile[2][kTileSteps];
    __shared__ __align__(8) uint64_t bar[2];

    const unsigned bid = blockIdx.x;
    const int p = (int)(bid % (unsigned)P.n_part);
    const unsigned rest = bid / (unsigned)P.n_part;
    const int cb = (int)(rest % (unsigned)P.n_cell_blocks);
    const int c = (int)(rest / (unsigned)P.n_cell_blocks);
    const int S = P.n_samples - 1;
    const int k_begin = P.k_first + c * P.chunk;
    const int k_end = min(S, k_begin + P.chunk - 1);
    const int n_int = k_end - k_begin + 1;
    const int n_tiles = (n_int + kTileSteps - 1) / kTileSteps;
    const RecD* rec = static_cast<const RecD*>(P.rec) + (size_t)p * P.n_samples;
    const int tid = threadIdx.x;
    const int cell = cb * kDepositThreads + tid;
    const bool active = cell < P.n_pix;

    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (tid == 0) {
        for (int t = 0; t < 2 && t < n_tiles; ++t) {
            const int k0 = k_begin + t * kTileSteps;
            const unsigned bytes = (unsigned)min(kTileSteps, k_end - k0 + 1) * sizeof(RecD);
            mbar_arrive_expect_tx(&bar[t], bytes);
            bulk_g2s(tile[t], rec + k0, bytes, &bar[t]);
        }
    }

    D64State st;
    D4 cl = {0.0, 0.0, 0.0, 0.0};
    double ncx = 0.0, ncy = 0.0, ncz = 1.0, Rc = 1.0;       // far-field limit: cell direction, distance
    const bool ff = P.ff != 0;
    bool live = false;
    double* row = nullptr;
    const double* xp = P.x + (size_t)p * P.n_samples * 3;
    if (active) {
        cl = P.cells[cell];
        double Ra, Re;
        const double* xa = xp + 3 * (size_t)(k_begin - 1);
        const double* xe = xp + 3 * (size_t)k_end;
        double ua, ue;
        if (ff) {
            farfield_cell(cl, ncx, ncy, ncz, Rc);
            ua = arrival_bins_ff(xa[0], xa[1], xa[2], ncx, ncy, ncz, Rc, cl.w, P.t0, k_begin - 1, P.dt, P.inv_dt_det);
            ue = arrival_bins_ff(xe[0], xe[1], xe[2], ncx, ncy, ncz, Rc, cl.w, P.t0, k_end, P.dt, P.inv_dt_det);
        } else {
            ua = arrival_bins(xa[0], xa[1], xa[2], cl, P.t0, k_begin - 1, P.dt, P.inv_dt_det, Ra);
            ue = arrival_bins(xe[0], xe[1], xe[2], cl, P.t0, k_end, P.dt, P.inv_dt_det, Re);
        }
        live = (ue > 0.0) && (ua < (double)P.n_bins);
        st.a = ua;
        st.b = clamp_bin(floor(ua));
        if (LM == 0) set_edge(st, (double)st.b + 1.0);
        st.n_below = (ua < 0.0) ? n_int : 0;
        st.n_above = 0;
#pragma unroll
        for (int i = 0; i < 6; ++i) st.acc[i] = 0.0;
        row = static_cast<double*>(P.fields) + (size_t)cell * P.n_bins * 6;
        if (!live) atomicAdd(&P.counters->clipped, (unsigned long long)n_int);
    }
    // held field: warps whose every lane walks a cell share their bin-start work (fp64_deposit_warp)
    const bool full_warp = LM == 0 && __ballot_sync(0xffffffffu, live) == 0xffffffffu;
    if (LM && live) {
        // field of the sample before the chunk; a trajectory's first interval holds F_1
        const RecD r0 = rec[k_begin > 1 ? k_begin - 1 : 1];
        if (ff) {
            fp64_field_ff(r0, ncx, ncy, ncz, Rc, st.Fp);
        } else {
            double dx, dy, dz, R0;
            (void)fp64_arrival(r0, cl, P.inv_dt_det, dx, dy, dz, R0);
            fp64_field(r0, dx, dy, dz, R0, st.Fp);
        }
        // RD_QUADRATIC: the field and arrival of the sample two before the chunk (used from the
        // trajectory's third interval on)
        st.ap = st.a - 1.0;
#pragma unroll
        for (int i = 0; i < 6; ++i) st.Fpp[i] = st.Fp[i];
        if (LM == 2 && k_begin >= 3) {
            const RecD r1 = rec[k_begin - 2];
            if (ff) {
                fp64_field_ff(r1, ncx, ncy, ncz, Rc, st.Fpp);
                st.ap = arrival_bins_ff(r1.xa.x, r1.xa.y, r1.xa.z, ncx, ncy, ncz, Rc, cl.w, P.t0, k_begin - 2, P.dt,
                                        P.inv_dt_det);
            } else {
                double dx, dy, dz, R1;
                st.ap = fp64_arrival(r1, cl, P.inv_dt_det, dx, dy, dz, R1);
                fp64_field(r1, dx, dy, dz, R1, st.Fpp);
            }
        }
    }

    for (int t = 0; t < n_tiles; ++t) {
        const int buf = t & 1;
        const bool ok = mbar_wait_bounded(&bar[buf], (unsigned)(t >> 1) & 1u);
        if (__syncthreads_or(!ok)) {
            if (tid == 0) {
                atomicOr(&P.counters->errors, ERRBIT_TIMEOUT);
                for (int u = t; u < t + 2 && u < n_tiles; ++u)
                    (void)mbar_wait_bounded(&bar[u & 1], (unsigned)(u >> 1) & 1u);
            }
            __syncthreads();
            return;
        }
        const int k0 = k_begin + t * kTileSteps;
        const int cnt = min(kTileSteps, k_end - k0 + 1);
        if (live) {
            double F[6];
            for (int i = 0; i < cnt; ++i) {
                const RecD r = tile[buf][i];
                const int k = k0 + i;
                double cbin;
                if (ff) {
                    fp64_field_ff(r, ncx, ncy, ncz, Rc, F);
                    cbin = arrival_bins_ff(r.xa.x, r.xa.y, r.xa.z, ncx, ncy, ncz, Rc, cl.w, P.t0, k, P.dt, P.inv_dt_det);
                } else {
                    double dx, dy, dz, R;
                    cbin = fp64_arrival(r, cl, P.inv_dt_det, dx, dy, dz, R);
                    fp64_field(r, dx, dy, dz, R, F);
                }
                if (LM) {
                    const double a_prev = st.a;
                    if (LM == 2 && k + P.k_real0 >= 3)
                        fp64_deposit_quad(st, F, cbin, row, P.n_bins, k, k_begin, k_end);
                    else    // RD_HOLD_PREV (lin 2): the previous field at both ends, i.e. held
                        fp64_deposit_lin(st, st.Fp, P.lin == 2 ? st.Fp : F, cbin, row, P.n_bins, k, k_begin, k_end);
#pragma unroll
                    for (int j = 0; j < 6; ++j) {
                        if (LM == 2) st.Fpp[j] = st.Fp[j];
                        st.Fp[j] = F[j];
                    }
                    if (LM == 2) st.ap = a_prev;
                } else {
                    if (full_warp)
                        fp64_deposit_warp(st, F, cbin, row, P.n_bins, k, k_begin, k_end);
                    else
                        fp64_deposit(st, F, cbin, row, P.n_bins, k, k_begin, k_end);
                }
            }
            if (t == n_tiles - 1) {
                flush_f64(row, P.n_bins, st.b, st.acc);
                const int clip = min(n_int, st.n_below + st.n_above);
                if (clip > 0) atomicAdd(&P.counters->clipped, (unsigned long long)clip);
            }
        }
        __syncthreads();
        if (tid == 0 && t + 2 < n_tiles) {
            fence_proxy_async();
            const int k2 = k_begin + (t + 2) * kTileSteps;
            const unsigned bytes = (unsigned)min(kTileSteps, k_end - k2 + 1) * sizeof(RecD);
            mbar_arrive_expect_tx(&bar[buf], bytes);
            bulk_g2s(tile[buf], rec + k2, bytes, &bar[buf]);
        }
    }
}

// =============================================================================================
// readout: internal layout -> E[n_pix][n_bins][3], B[n_pix][n_bins][3]
// =============================================================================================
template <typename Tin, int STRIDE, typename Tout>
__global__ void k_read(const Tin* __restrict__ fields, long long n, Tout* __restrict__ E,
                       Tout* __restrict__ B)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const Tin* v = fields + i * STRIDE;
        if (E) {
            E[3 * i] = (Tout)v[0];
            E[3 * i + 1] = (Tout)v[1];
            E[3 * i + 2] = (Tout)v[2];
        }
        if (B) {
            B[3 * i] = (Tout)v[3];
            B[3 * i + 1] = (Tout)v[4];
            B[3 * i + 2] = (Tout)v[5];
        }
    }
}

// E[n_pix][n_bins][3], B[...] -> internal layout (the inverse of k_read); a NULL E or B sets that
// part to zero, and the padding of the mixed layout is cleared
template <typename Tin, int STRIDE, typename Tf>
__global__ void k_write(Tf* __restrict__ fields, long long n, const Tin* __restrict__ E, const Tin* __restrict__ B)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        Tf* v = fields + i * STRIDE;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            v[c] = E ? (Tf)E[3 * i + c] : (Tf)0;
            v[3 + c] = B ? (Tf)B[3 * i + c] : (Tf)0;
        }
#pragma unroll
        for (int c = 6; c < STRIDE; ++c) v[c] = (Tf)0;
    }
}

// =============================================================================================
// launchers
// =============================================================================================
static int grid_for(long long n, int threads) { return grid_stride_blocks(n, threads, 16); }

cudaError_t launch_precompute_mixed(const double* x, const double* u, const double* q, double qscale, int n_part,
                                    int n_samples, double dt, int flags, RecS* rec, DevCounters* counters,
                                    cudaStream_t s)
{
    const long long n = (long long)n_part * n_samples;
    const PrecomputeGrid g(n);
    k_precompute_mixed<<<g.blocks, g.threads, 0, s>>>(x, u, q, qscale, n, n_samples, dt, flags, rec, counters);
    return cudaGetLastError();
}

cudaError_t launch_precompute_fp64(const double* x, const double* u, const double* q, int n_part, int n_samples,
                                   double t0, double dt, int flags, RecD* rec, DevCounters* counters, cudaStream_t s)
{
    const long long n = (long long)n_part * n_samples;
    const PrecomputeGrid g(n);
    k_precompute_fp64<<<g.blocks, g.threads, 0, s>>>(x, u, q, n, n_samples, t0, dt, flags, rec, counters);
    return cudaGetLastError();
}

cudaError_t launch_deposit_fp64(const DepositParams& p, int flags, cudaStream_t s)
{
    const long long blocks = (long long)p.n_cell_blocks * p.n_part * p.n_chunks;
    if (blocks <= 0) return cudaSuccess;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    if (p.lin == 3)
        k_deposit_fp64<2><<<(unsigned)blocks, kDepositThreads, 0, s>>>(p, flags);
    else if (p.lin)
        k_deposit_fp64<1><<<(unsigned)blocks, kDepositThreads, 0, s>>>(p, flags);
    else
        k_deposit_fp64<0><<<(unsigned)blocks, kDepositThreads, 0, s>>>(p, flags);
    return cudaGetLastError();
}

cudaError_t launch_read_fields(const void* fields, int precision, int n_pix, int n_bins, void* E,
                               void* B, int dtype, cudaStream_t s)
{
    const long long n = (long long)n_pix * n_bins;
    const int g = grid_for(n, 256);
    if (precision == RD_MIXED) {
        if (dtype == RD_F32)
            k_read<float, 8, float><<<g, 256, 0, s>>>(static_cast<const float*>(fields), n,
                                                      static_cast<float*>(E), static_cast<float*>(B));
        else
            k_read<float, 8, double><<<g, 256, 0, s>>>(static_cast<const float*>(fields), n,
                                                       static_cast<double*>(E), static_cast<double*>(B));
    } else {
        if (dtype == RD_F32)
            k_read<double, 6, float><<<g, 256, 0, s>>>(static_cast<const double*>(fields), n,
                                                       static_cast<float*>(E), static_cast<float*>(B));
        else
            k_read<double, 6, double><<<g, 256, 0, s>>>(static_cast<const double*>(fields), n,
                                                        static_cast<double*>(E), static_cast<double*>(B));
    }
    return cudaGetLastError();
}

cudaError_t launch_write_fields(void* fields, int precision, int n_pix, int n_bins, const void* E, const void* B,
                                int dtype, cudaStream_t s)
{
    const long long n = (long long)n_pix * n_bins;
    const int g = grid_for(n, 256);
    if (precision == RD_MIXED) {
        if (dtype == RD_F32)
            k_write<float, 8, float><<<g, 256, 0, s>>>(static_cast<float*>(fields), n, static_cast<const float*>(E),
                                                       static_cast<const float*>(B));
        else
            k_write<double, 8, float><<<g, 256, 0, s>>>(static_cast<float*>(fields), n, static_cast<const double*>(E),
                                                        static_cast<const double*>(B));
    } else {
        if (dtype == RD_F32)
            k_write<float, 6, double><<<g, 256, 0, s>>>(static_cast<double*>(fields), n, static_cast<const float*>(E),
                                                        static_cast<const float*>(B));
        else
            k_write<double, 6, double><<<g, 256, 0, s>>>(static_cast<double*>(fields), n,
                                                         static_cast<const double*>(E), static_cast<const double*>(B));
    }
    return cudaGetLastError();
}

}  // namespace rd
