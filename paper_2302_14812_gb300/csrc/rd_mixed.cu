// Mixed-precision deposit: FP32 Lienard-Wiechert field (Eq. 1) and FP32 accumulation, with the
// arrival time (Eq. 2) kept FP64-accurate.
//
// Work item = (step chunk, block of CPC cells, particle) with CPC = 64, 128 or 256 (the launch
// shape; 256 by default), ordered by item_coords: consecutive CTAs take one particle to a small
// group of cell blocks, then the next particle (odd groups in reverse particle order), so the CTAs
// resident at one time reduce into the group's slice of the detector, which stays in L2, and each
// particle's staged records come from DRAM about once per group.
//
// Each thread walks NC cells (1 or 2) through the chunk; the per-sample constants (RecS) are read
// once per sample from shared memory and serve all of them.  Per cell the walk carries the bin it
// is filling (as an offset from the CTA's first field row) and the time f already spent in that
// bin, in units of dt; a step adds the arrival-time increment
//     t'_k - t'_{k-1} = dt [dt g + R_k (g + |n_k - vbar|^2)] / (dt + R_k + R_{k-1})
// (vbar = (x_k - x_{k-1})/dt, g = 1 - |vbar|^2), an exact identity with only positive terms, so
// FP32 keeps its relative precision; the chunk's first and last arrival times are computed in
// FP64 directly from Eq. 2 (anchors), which bounds the drift to one chunk and makes adjacent
// chunks meet exactly.  The field held over the interval is added to the running bin with the
// part of the interval that lies in that bin (integrating deposit, Section 3.2); when the arrival
// time leaves the bin, the bin is added to global memory with two vector reductions.
#include <math.h>

#include <algorithm>

#include "rd_internal.cuh"

namespace rd {

namespace {

// Bin indices of the walk are clamped to +-2^29 so that offsets (row * n_bins + bin, with
// n_bins <= kMixedMaxBins) and differences of two of them stay inside int32.
constexpr double kWalkClamp = 536870912.0;

__device__ __forceinline__ int walk_bin(double fb) { return (int)fmin(fmax(fb, -kWalkClamp), kWalkClamp); }

// Walk state of the thread's NC cells.
template <int NC>
struct Cells {
    float px[NC], py[NC], pz[NC];   // cell positions
    float f[NC];                    // time spent in the current bin, units of dt (0 <= f < W)
    float rpd[NC];                  // R_{k-1} + dt (far-field limit: 1/R_c)
    float nlx[NC], nly[NC], nlz[NC];  // far-field limit: n_c - (its FP32 rounding in px, py, pz)
    float acc[6][NC];               // E xyz, B xyz of the current bin so far (weights in bins)
    int bo[NC];                     // row * n_bins + bin being filled (bin may lie outside the window)
};

// What a cell needs only at the ends of its chunk, kept in shared memory ([word][thread]) so that the
// walk's registers hold nothing but its running state.
enum { kBoEnd, kFEnd, kBelow, kAbove, kColdWords };
template <int NC, int NT>
struct Cold {
    float (*w)[NT];                 // [NC * kColdWords][NT]
    // row * n_bins + bin, and time inside that bin, of the chunk's last arrival (exact FP64 anchor)
    __device__ __forceinline__ int bo_end(int j) const { return __float_as_int(w[j * kColdWords + kBoEnd][threadIdx.x]); }
    __device__ __forceinline__ float f_end(int j) const { return w[j * kColdWords + kFEnd][threadIdx.x]; }
    // intervals whose start lies before / whose end lies after the window; below = -1: a cell without
    // arrivals in the window
    __device__ __forceinline__ int below(int j) const { return __float_as_int(w[j * kColdWords + kBelow][threadIdx.x]); }
    __device__ __forceinline__ int above(int j) const { return __float_as_int(w[j * kColdWords + kAbove][threadIdx.x]); }
    __device__ __forceinline__ void set(int j, int word, int v) const { w[j * kColdWords + word][threadIdx.x] = __int_as_float(v); }
    __device__ __forceinline__ void set(int j, int word, float v) const { w[j * kColdWords + word][threadIdx.x] = v; }
};

// Offset of cell row j's first bin: row * n_bins (row = the cell's index inside the CTA's block).
template <int NT>
__device__ __forceinline__ int row_base(int j, int n_bins) { return (j * NT + (int)threadIdx.x) * n_bins; }

#ifndef RD_CHECK
#define RD_CHECK 0   // 1: the walk's unguarded reductions check their bin (a checked build, for tests)
#endif

struct Consts {
    float W;                        // bin width / dt
    float invW;
    float DT;
    int n_bins;
    float* base;                    // field row 0 of the CTA's cell block
    int kq;                         // quadratic interpolation: first interval (this call's index) with
                                    // three fields behind it (the trajectory's third interval)
#if RD_CHECK
    unsigned* errors;               // the detector's latched error bits
#endif
};

// Checked build: a reduction the window margin should keep inside the detector row is verified,
// and one that would leave it latches RD_ERR_BOUNDS and is dropped.
__device__ __forceinline__ bool bin_ok(const Consts& C, int b)
{
#if RD_CHECK
    if ((unsigned)b < (unsigned)C.n_bins) return true;
    atomicOr(C.errors, ERRBIT_BOUNDS);
    return false;
#else
    (void)C;
    (void)b;
    return true;
#endif
}

// Field of one sample at one cell, scaled to the bin weights (E = S E', B = (S/R) d x E').
struct Field {
    float E[3];                     // E' = Q [(n - beta)(-c1/kappa) + betadot],  Q = -q dt/dt_det
    float B[3];                     // d x E'
    float S;                        // 1 / (kappa^2 R)
    float rinv;                     // 1 / R
    float num, rden;                // t'_k - t'_{k-1} = num * rden in units of dt
};

__device__ __forceinline__ float* bin_addr(const Consts& C, int bo)
{
    return reinterpret_cast<float*>(reinterpret_cast<char*>(C.base) + (size_t)(unsigned)bo * 32u);
}

// Add one bin (b = bin index, bo = its offset) to global memory; bins outside the window are dropped.
__device__ __forceinline__ void flush(const Consts& C, int b, int bo, float e0, float e1, float e2, float b0,
                                      float b1, float b2)
{
    if ((unsigned)b < (unsigned)C.n_bins) {
        float* p = bin_addr(C, bo);
        red_add_v4(p, e0, e1, e2, b0);
        red_add_v2(p + 4, b1, b2);
    }
}

// B of a bin.  Far-field limit: every sample of a cell has the same n_c and scale (1/R_c folded
// into S, 1/R = 1), so B = n_c x E holds for each sample's weighted field and hence for the bin
// sums: the walk carries E only and forms B when the bin is written.  Otherwise B is carried.
template <int NC, bool FF>
__device__ __forceinline__ void bin_b(const Cells<NC>& c, int j, const float* e, const float* carried, float* b)
{
    if (FF) {
        b[0] = fmaf(c.py[j], e[2], -(c.pz[j] * e[1]));
        b[1] = fmaf(c.pz[j], e[0], -(c.px[j] * e[2]));
        b[2] = fmaf(c.px[j], e[1], -(c.py[j] * e[0]));
    } else {
        b[0] = carried[0];
        b[1] = carried[1];
        b[2] = carried[2];
    }
}

// Add bin b of cell j from its accumulator.
template <int NC, bool FF>
__device__ __forceinline__ void flush_acc(const Consts& C, const Cells<NC>& c, int j, int b, int bo)
{
    const float e[3] = {c.acc[0][j], c.acc[1][j], c.acc[2][j]};
    const float cb[3] = {c.acc[3][j], c.acc[4][j], c.acc[5][j]};
    float bb[3];
    bin_b<NC, FF>(c, j, e, cb, bb);
    flush(C, b, bo, e[0], e[1], e[2], bb[0], bb[1], bb[2]);
}

// Eq. 1 with B = n x E at one cell:
//   E = q/(kappa^3 R) [ (n - beta)(gamma^-2/R + n.betadot) - betadot kappa ]
//     = S E',  S = 1/(kappa^2 R),  E' = -q [(n - beta)(-c1/kappa) + betadot],  c1 = gamma^-2/R + n.betadot
//   B = n x E = (S/R) d x E'
// E' also carries the bin weight per unit dt (the records hold Q = -q dt/dt_det times betadot and
// gamma^-2), and kappa = (gamma^-2 + |n - beta|^2)/2 avoids the cancellation in 1 - beta.n.
__device__ __forceinline__ void field_at(const RecS& r, float px, float py, float pz, float& rpd, const Consts& C,
                                         Field& o)
{
    // geometry: d = x_cell - x_k, R = |d|
    const float dx = px + r.nx, dy = py + r.ny, dz = pz + r.nz;
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const float rinv = fast_rsqrt(r2);
    const float bx = fmaf(dx, rinv, r.nbx), by = fmaf(dy, rinv, r.nby), bz = fmaf(dz, rinv, r.nbz);   // n - beta
    const float nb2 = fmaf(bx, bx, fmaf(by, by, bz * bz));
    // arrival-time increment in units of dt, numerator and denominator divided by R:
    //   [dt g / R + (g + |n - vbar|^2)] / [1 + (R_{k-1} + dt) / R],
    //   g + |n - vbar|^2 = |n - beta|^2 + 2 (n - beta).(beta - vbar) + (g + |beta - vbar|^2)
    const float gg = fmaf(bx, r.d2x, fmaf(by, r.d2y, fmaf(bz, r.d2z, nb2 + r.gd)));
    const float num = fmaf(r.dtg, rinv, gg);
    const float den = fmaf(rpd, rinv, 1.f);
    o.num = num;
    o.rden = fast_rcp(den);
    rpd = fmaf(r2, rinv, C.DT);
    // Eq. 1
    const float kn = fmaf(nb2, -0.5f, r.nhig2);                         // -kappa
    const float ikn = fast_rcp(kn);                                     // -1/kappa
    const float nrik = rinv * ikn;                                      // -1/(kappa R)
    o.S = nrik * ikn;                                                   // 1/(kappa^2 R)
    // with the record's charge factor Q: Q (gamma^-2 + d.betadot) (-1/(kappa R)) = -Q c1/kappa
    const float c1n = fmaf(dx, r.bdx, fmaf(dy, r.bdy, fmaf(dz, r.bdz, r.ig2n))) * nrik;
    o.E[0] = fmaf(bx, c1n, r.bdx);
    o.E[1] = fmaf(by, c1n, r.bdy);
    o.E[2] = fmaf(bz, c1n, r.bdz);
    o.B[0] = fmaf(dy, o.E[2], -(dz * o.E[1]));
    o.B[1] = fmaf(dz, o.E[0], -(dx * o.E[2]));
    o.B[2] = fmaf(dx, o.E[1], -(dy * o.E[0]));
    o.rinv = rinv;
}

// Far-field limit (RD_FARFIELD) at one cell, seen from the origin along n_c at R_c (n_c and
// 1/R_c fixed per cell):
//   t'_k - t'_{k-1} = dt (1 - n_c.vbar) = dt [g + |n_c - vbar|^2] / 2   (Eq. 3, |n_c| = 1)
//   E = S E',  S = 1/(kappa^2 R_c),  E' = Q [(n_c - beta)(-n_c.betadot/kappa) + betadot],  B = S n_c x E'
// with kappa = 1 - beta.n_c = (gamma^-2 + |n_c - beta|^2)/2.  n_c is held as its FP32 rounding
// (nx, ny, nz) plus the rest (lx, ly, lz): the rounding is fixed per cell, and along the beam, where
// n_c - beta is ~1e-3, it would bias kappa by ~5e-5 (the field by ~1.5e-4, as kappa^-3) on every
// sample of the cell.  nx - beta_x is exact there (the two are within a factor of two), and adding
// the rest restores n_c - beta to FP32 precision.
__device__ __forceinline__ void field_at_ff(const RecS& r, float nx, float ny, float nz, float invR, float lx,
                                            float ly, float lz, Field& o)
{
    const float bx = (nx + r.nbx) + lx, by = (ny + r.nby) + ly, bz = (nz + r.nbz) + lz;   // n_c - beta
    const float nb2 = fmaf(bx, bx, fmaf(by, by, bz * bz));
    o.num = fmaf(bx, r.d2x, fmaf(by, r.d2y, fmaf(bz, r.d2z, nb2 + r.gd)));
    o.rden = 0.5f;
    const float kn = fmaf(nb2, -0.5f, r.nhig2);                         // -kappa
    const float ikn = fast_rcp(kn);
    o.S = (ikn * ikn) * invR;
    const float c1n = fmaf(nx, r.bdx, fmaf(ny, r.bdy, nz * r.bdz)) * ikn; // -Q n_c.betadot / kappa
    o.E[0] = fmaf(bx, c1n, r.bdx);
    o.E[1] = fmaf(by, c1n, r.bdy);
    o.E[2] = fmaf(bz, c1n, r.bdz);
    o.B[0] = fmaf(ny, o.E[2], -(nz * o.E[1]));
    o.B[1] = fmaf(nz, o.E[0], -(nx * o.E[2]));
    o.B[2] = fmaf(nx, o.E[1], -(ny * o.E[0]));
    o.rinv = 1.f;
}

// The walk of a tile.  The fast walk has no code for an interval that passes two or more bin edges; such an
// interval sets the cell's time to -inf, after which the cell crosses no edge and flushes nothing for the
// rest of the tile.  The exact walk handles any interval.  It walks a tile again (from its saved start)
// for a warp in which some cell stopped, flushing only from the interval that stopped it onwards (earlier
// bins were flushed by the fast walk), and then walks that warp's next tile at once.  Both evaluate the
// arrival times with the same operations in the same order (no implicit contraction), so they agree bit
// for bit up to that interval.

// Fast step: one interval for all cells of the thread: field of the sample (Eq. 1), the part of
// [f, f + du] inside the current bin added to the running bin; a cell whose arrival time passes the bin
// edge flushes the bin and starts the next one with the rest of the interval.  LAST: the interval ends
// on the exact FP64 anchors.  TRACK: bins may lie outside the window (checked, clipped intervals
// counted).
template <int NC, int NT, bool LAST, bool TRACK, bool FF>
__device__ __forceinline__ void step(Cells<NC>& c, const RecS& r, const Consts& C, const Cold<NC, NT>& cold, int k,
                                     int k_begin, int k_end)
{
    Field o[NC];
    float fn[NC];
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        if (FF)
            field_at_ff(r, c.px[j], c.py[j], c.pz[j], c.rpd[j], c.nlx[j], c.nly[j], c.nlz[j], o[j]);
        else
            field_at(r, c.px[j], c.py[j], c.pz[j], c.rpd[j], C, o[j]);
        float t;
        if (LAST) {
            t = fmaf((float)(cold.bo_end(j) - c.bo[j]), C.W, cold.f_end(j));
            t = c.f[j] == -INFINITY ? -INFINITY : t;
        } else {
            t = fmaf(o[j].num, o[j].rden, c.f[j]);
        }
        const float ws = (fminf(t, C.W) - c.f[j]) * o[j].S;
        const float wb = ws * o[j].rinv;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            c.acc[i][j] = fmaf(o[j].E[i], ws, c.acc[i][j]);
            if (!FF) c.acc[3 + i][j] = fmaf(o[j].B[i], wb, c.acc[3 + i][j]);
        }
        fn[j] = t < 2.f * C.W ? t : -INFINITY;
    }
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        // the arrival time passed the bin edge (a time exactly on the edge belongs to the upper bin)
        const bool cr = fn[j] >= C.W;
        c.f[j] = fn[j];
        if (cr) {
            const int b = TRACK || RD_CHECK ? c.bo[j] - row_base<NT>(j, C.n_bins) : 0;
            const float e[3] = {c.acc[0][j], c.acc[1][j], c.acc[2][j]};
            const float cb[3] = {c.acc[3][j], c.acc[4][j], c.acc[5][j]};
            float bb[3];
            bin_b<NC, FF>(c, j, e, cb, bb);
            if (TRACK ? (unsigned)b < (unsigned)C.n_bins : (!RD_CHECK || bin_ok(C, b))) {
                float* a = bin_addr(C, c.bo[j]);
                red_add_v4(a, e[0], e[1], e[2], bb[0]);
                red_add_v2(a + 4, bb[1], bb[2]);
            }
            const float rem = fn[j] - C.W;
            const float rs = rem * o[j].S;
            const float rbw = rs * o[j].rinv;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                c.acc[i][j] = o[j].E[i] * rs;
                if (!FF) c.acc[3 + i][j] = o[j].B[i] * rbw;
            }
            c.f[j] = rem;
            c.bo[j] += 1;
            if (TRACK) {
                if (b == -1) cold.set(j, kBelow, k - k_begin + 1);
                if (b == C.n_bins - 1) cold.set(j, kAbove, k_end - k + 1);
            }
        }
    }
}

#ifndef RD_UNROLL
#define RD_UNROLL 0
#endif
constexpr int kUnroll = RD_UNROLL > 0 ? RD_UNROLL : 1;   // samples per loop iteration

// ---------------------------------------------------------------------------------------------
// Two cells per thread as packed pairs, two intervals at a time (the unchecked walk of the held field).
//
// What bounds the walk is the register file: a three-operand FP32 instruction whose operands are all
// different registers takes 1.7 issue cycles on this part (1.2 with two operands reused; measured with
// independent chains), so the scalar step's 74 instructions per 32 (cell, interval) pairs read about
// 165 registers and ran at 93 cycles, 0.8 of the issue slots.  Two-wide instructions (fma.rn.f32x2 and
// its kin, rounded like the scalar ones) read a sample's constant once for both cells, and two intervals
// per crossing update halve its reductions, branches and addressing: 53 instructions and 87 cycles.
// Measured on 1000 electrons x 4000 steps x 16384 cells x 2048 bins: 149.9 -> 139.4 ms per launch (139.8 now); two
// cells packed, one interval at a time: 154.4 ms; accumulators packed as well: 141.7 ms (their halves
// are written one by one on a crossing, which costs a copy of every accumulator per pass); one crossing
// update for both cells with selects: 155 ms.  128 registers (4 CTAs of 128 threads per SM) rather than
// 96 (5 CTAs: 143.4 ms with packed accumulators).
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    float2 d;
    asm("{\n\t.reg .b64 A, B, C, D;\n\tmov.b64 A, {%2, %3};\n\tmov.b64 B, {%4, %5};\n\tmov.b64 C, {%6, %7};\n\t"
        "fma.rn.ftz.f32x2 D, A, B, C;\n\tmov.b64 {%0, %1}, D;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}

__device__ __forceinline__ float2 mul2(float2 a, float2 b)
{
    float2 d;
    asm("{\n\t.reg .b64 A, B, D;\n\tmov.b64 A, {%2, %3};\n\tmov.b64 B, {%4, %5};\n\t"
        "mul.rn.ftz.f32x2 D, A, B;\n\tmov.b64 {%0, %1}, D;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}

__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    float2 d;
    asm("{\n\t.reg .b64 A, B, D;\n\tmov.b64 A, {%2, %3};\n\tmov.b64 B, {%4, %5};\n\t"
        "add.rn.ftz.f32x2 D, A, B;\n\tmov.b64 {%0, %1}, D;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}

__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    float2 d;
    asm("{\n\t.reg .b64 A, B, D;\n\tmov.b64 A, {%2, %3};\n\tmov.b64 B, {%4, %5};\n\t"
        "sub.rn.ftz.f32x2 D, A, B;\n\tmov.b64 {%0, %1}, D;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 rcp2(float2 a) { return make_float2(fast_rcp(a.x), fast_rcp(a.y)); }
__device__ __forceinline__ float2 pair_of(const float (&v)[2]) { return make_float2(v[0], v[1]); }
__device__ __forceinline__ void set_pair(float (&v)[2], float2 a)
{
    v[0] = a.x;
    v[1] = a.y;
}

struct Field2 {
    float2 E[3], B[3], S, rinv, num, rden;      // as Field, for both cells (far-field limit: B, rinv unused)
};

// field_at / field_at_ff for the two cells, with the same operations in the same order.
template <bool FF>
__device__ __forceinline__ void field_pair(const RecS& r, Cells<2>& c, const Consts& C, Field2& o)
{
    if (FF) {
        const float2 nx = pair_of(c.px), ny = pair_of(c.py), nz = pair_of(c.pz);
        const float2 bx = add2(add2(nx, both(r.nbx)), pair_of(c.nlx)), by = add2(add2(ny, both(r.nby)), pair_of(c.nly)),
                     bz = add2(add2(nz, both(r.nbz)), pair_of(c.nlz));
        const float2 nb2 = fma2(bx, bx, fma2(by, by, mul2(bz, bz)));
        o.num = fma2(bx, both(r.d2x), fma2(by, both(r.d2y), fma2(bz, both(r.d2z), add2(nb2, both(r.gd)))));
        o.rden = both(0.5f);
        const float2 ikn = rcp2(fma2(nb2, both(-0.5f), both(r.nhig2)));
        o.S = mul2(mul2(ikn, ikn), pair_of(c.rpd));
        const float2 c1n = mul2(fma2(nx, both(r.bdx), fma2(ny, both(r.bdy), mul2(nz, both(r.bdz)))), ikn);
        o.E[0] = fma2(bx, c1n, both(r.bdx));
        o.E[1] = fma2(by, c1n, both(r.bdy));
        o.E[2] = fma2(bz, c1n, both(r.bdz));
        return;
    }
    const float2 dx = add2(pair_of(c.px), both(r.nx)), dy = add2(pair_of(c.py), both(r.ny)),
                 dz = add2(pair_of(c.pz), both(r.nz));
    const float2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
    const float2 rinv = make_float2(fast_rsqrt(r2.x), fast_rsqrt(r2.y));
    const float2 bx = fma2(dx, rinv, both(r.nbx)), by = fma2(dy, rinv, both(r.nby)), bz = fma2(dz, rinv, both(r.nbz));
    const float2 nb2 = fma2(bx, bx, fma2(by, by, mul2(bz, bz)));
    const float2 gg = fma2(bx, both(r.d2x), fma2(by, both(r.d2y), fma2(bz, both(r.d2z), add2(nb2, both(r.gd)))));
    o.num = fma2(both(r.dtg), rinv, gg);
    o.rden = rcp2(fma2(pair_of(c.rpd), rinv, both(1.f)));
    set_pair(c.rpd, fma2(r2, rinv, both(C.DT)));
    const float2 kn = fma2(nb2, both(-0.5f), both(r.nhig2));
    const float2 ikn = rcp2(kn);
    const float2 nrik = mul2(rinv, ikn);
    o.S = mul2(nrik, ikn);
    const float2 c1n = mul2(fma2(dx, both(r.bdx), fma2(dy, both(r.bdy), fma2(dz, both(r.bdz), both(r.ig2n)))), nrik);
    o.E[0] = fma2(bx, c1n, both(r.bdx));
    o.E[1] = fma2(by, c1n, both(r.bdy));
    o.E[2] = fma2(bz, c1n, both(r.bdz));
    // d x E'; the negated products are written as 0 - product, which the subtraction absorbs (a sign
    // flip of each half would be two more instructions)
    const float2 zero = both(0.f);
    o.B[0] = fma2(dy, o.E[2], sub2(zero, mul2(dz, o.E[1])));
    o.B[1] = fma2(dz, o.E[0], sub2(zero, mul2(dx, o.E[2])));
    o.B[2] = fma2(dx, o.E[1], sub2(zero, mul2(dy, o.E[0])));
    o.rinv = rinv;
}

// acc += weight (per unit S) times the field, both cells.
template <bool FF>
__device__ __forceinline__ void add_field(Cells<2>& c, const Field2& o, float2 w)
{
    const float2 ws = mul2(w, o.S), wb = FF ? ws : mul2(ws, o.rinv);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        c.acc[i][0] = fmaf(o.E[i].x, ws.x, c.acc[i][0]);
        c.acc[i][1] = fmaf(o.E[i].y, ws.y, c.acc[i][1]);
        if (!FF) {
            c.acc[3 + i][0] = fmaf(o.B[i].x, wb.x, c.acc[3 + i][0]);
            c.acc[3 + i][1] = fmaf(o.B[i].y, wb.y, c.acc[3 + i][1]);
        }
    }
}

__device__ __forceinline__ float half_of(float2 a, int j) { return j == 0 ? a.x : a.y; }
__device__ __forceinline__ void set_half(float2& a, int j, float v)
{
    if (j == 0) a.x = v;
    else a.y = v;
}

// What a walk does about the ends of the window: nothing (every bin it passes lies inside), check and count where
// an edge is passed, or either by a flag read there.
enum : int { kUntracked, kTracked, kTrackFlag };

// Where the walk stands in the chunk (for the counts of clipped intervals).
struct Place {
    int k, k_begin, k_end;
    bool track;
};

// Cell j's arrival time passes the edge of the bin it is filling, in interval k: add that bin to global memory.
// Untracked, the bin is inside the window; tracked, it is checked and the crossings of the window's ends are noted.
template <int NT, bool FF, int TRACK>
__device__ __forceinline__ void red_bin(const Consts& C, const Cells<2>& c, int j, const Cold<2, NT>& cold, const Place& at,
                                        int k)
{
    if (TRACK == kTracked || (TRACK == kTrackFlag && at.track)) {
        const int b = c.bo[j] - row_base<NT>(j, C.n_bins);
        if (b == -1) cold.set(j, kBelow, k - at.k_begin + 1);
        if (b == C.n_bins - 1) cold.set(j, kAbove, at.k_end - k + 1);
        if ((unsigned)b >= (unsigned)C.n_bins) return;
    } else if (RD_CHECK && !bin_ok(C, c.bo[j] - row_base<NT>(j, C.n_bins))) {
        return;
    }
    float* a = bin_addr(C, c.bo[j]);
    const float e[3] = {c.acc[0][j], c.acc[1][j], c.acc[2][j]};
    const float cb[3] = {c.acc[3][j], c.acc[4][j], c.acc[5][j]};
    float b[3];
    bin_b<2, FF>(c, j, e, cb, b);
    red_add_v4(a, e[0], e[1], e[2], b[0]);
    red_add_v2(a + 4, b[1], b[2]);
}

// The deposit of one interval (the fast step) from the fields of its sample.
template <int NT, bool FF, int TRACK>
__device__ __forceinline__ void deposit_pair(Cells<2>& c, const Field2& o, const Consts& C, const Cold<2, NT>& cold,
                                             const Place& at, int k)
{
    const float2 t = fma2(o.num, o.rden, pair_of(c.f));
    add_field<FF>(c, o, sub2(make_float2(fminf(t.x, C.W), fminf(t.y, C.W)), pair_of(c.f)));
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        float fn = half_of(t, j);
        fn = fn < 2.f * C.W ? fn : -INFINITY;
        c.f[j] = fn;
        if (fn >= C.W) {
            red_bin<NT, FF, TRACK>(C, c, j, cold, at, k);
            const float rem = fn - C.W;
            const float rs = rem * half_of(o.S, j), rbw = FF ? rs : rs * half_of(o.rinv, j);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                c.acc[i][j] = half_of(o.E[i], j) * rs;
                if (!FF) c.acc[3 + i][j] = half_of(o.B[i], j) * rbw;
            }
            c.f[j] = rem;
            c.bo[j] += 1;
        }
    }
}

// Two intervals (samples ra, then rb) at once.  A cell whose two intervals pass at most one bin edge
// needs one crossing update for both: the bin being filled takes the parts of both intervals below the
// edge, is flushed, and the next bin starts with the parts above it.  The arrival times and bins equal
// those of two single steps bit for bit (the exact re-walk of a tile relies on it).  A warp with a cell
// that passes two edges takes the two single steps instead.
template <int NT, bool FF, int TRACK>
__device__ __forceinline__ void two_steps_pair(Cells<2>& c, const RecS& ra, const RecS& rb, const Consts& C,
                                               const Cold<2, NT>& cold, const Place& at)
{
    Field2 a, b;
    field_pair<FF>(ra, c, C, a);
    field_pair<FF>(rb, c, C, b);
    const float2 t1 = fma2(a.num, a.rden, pair_of(c.f));
    const bool c1x = t1.x >= C.W, c1y = t1.y >= C.W;            // the first interval passes the edge
    const float2 r1 = add2(t1, both(-C.W));
    const float2 f1 = make_float2(c1x ? r1.x : t1.x, c1y ? r1.y : t1.y);
    const float2 t2 = fma2(b.num, b.rden, f1);
    // false for a NaN too (the single steps stop such a cell)
    const bool ok = t2.x < (c1x ? C.W : 2.f * C.W) && t2.y < (c1y ? C.W : 2.f * C.W);
    if (!__all_sync(0xffffffffu, ok)) {
        deposit_pair<NT, FF, TRACK>(c, a, C, cold, at, at.k);
        deposit_pair<NT, FF, TRACK>(c, b, C, cold, at, at.k + 1);
        return;
    }
    const float2 m1 = make_float2(fminf(t1.x, C.W), fminf(t1.y, C.W));
    const float2 m2 = make_float2(fminf(t2.x, C.W), fminf(t2.y, C.W));
    const float2 wf = sub2(m2, f1);
    add_field<FF>(c, a, sub2(m1, pair_of(c.f)));
    add_field<FF>(c, b, make_float2(c1x ? 0.f : wf.x, c1y ? 0.f : wf.y));
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const bool c1 = j == 0 ? c1x : c1y;
        const float tt = half_of(t2, j);
        c.f[j] = tt;
        if (c1 || tt >= C.W) {
            red_bin<NT, FF, TRACK>(C, c, j, cold, at, c1 ? at.k : at.k + 1);
            const float r2 = tt - C.W;
            const float wa = c1 ? half_of(r1, j) : 0.f;
            const float wb = c1 ? half_of(wf, j) : r2;
            const float sa = wa * half_of(a.S, j), sb = wb * half_of(b.S, j);
            const float ba = FF ? sa : sa * half_of(a.rinv, j), bb = FF ? sb : sb * half_of(b.rinv, j);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                c.acc[i][j] = fmaf(half_of(b.E[i], j), sb, half_of(a.E[i], j) * sa);
                if (!FF) c.acc[3 + i][j] = fmaf(half_of(b.B[i], j), bb, half_of(a.B[i], j) * ba);
            }
            c.f[j] = c1 ? tt : r2;
            c.bo[j] += 1;
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Interpolated fields (two cells per thread as packed pairs).
//
// RD_LINEAR: over interval k (length L, arrival times f to f + L) the field goes linearly from F_{k-1} to
// F_k, so the part [s0, s1] of the interval weighs F_{k-1} with (s1 - s0) - ramp and F_k with
// ramp = (s1^2 - s0^2) / (2 L).  RD_HOLD_PREV is the same walk with the ramps scaled to zero.
// RD_QUADRATIC adds D2 cu, D2 the second divided difference of F_{k-2}, F_{k-1}, F_k over their arrival
// times (spacings h and L) and cu = int_{s0}^{s1} s (s - L) ds: weights cu alpha on F_k,
// -cu (alpha + beta) on F_{k-1}, cu beta on F_{k-2}, alpha = 1 / (L (L + h)), beta = 1 / (h (L + h)).
//
// A sample's field so enters a bin with weights from two (three) intervals.  The walk does not add it once
// per interval: it carries the weight that is still to come (Prev::r) and adds a field to the running bin
// when its last interval is known, or when a bin ends in between.  That is one accumulation per interval
// as for the held field, instead of two (three, and the differences that D2 is made of).  Measured on 200
// electrons x 4000 steps x 16384 cells x 2048 bins: linear 43.6 -> 35.7 ms, quadratic 63.7 -> 50.8 ms (a bin edge
// passed in 18 % of the steps).
// ---------------------------------------------------------------------------------------------
struct Prev {                       // an earlier sample's field at both cells
    float2 E[3], B[3], S, SB;       // E = S E', B = SB (d x E') (far-field limit: B unused)
    float2 r;                       // weight of the running bin still to be added
};

struct LinState {
    Prev p1, p2;                    // samples k-1 and (quadratic) k-2
    float2 h;                       // quadratic: length of interval k-1
};

// int_0^s t (t - L) dt
__device__ __forceinline__ float qcube(float s, float L) { return (s * s) * fmaf(s, 1.f / 3.f, -0.5f * L); }
__device__ __forceinline__ float2 qcube2(float2 s, float2 L)
{
    return mul2(mul2(s, s), fma2(s, both(1.f / 3.f), mul2(both(-0.5f), L)));
}

template <bool FF>
__device__ __forceinline__ void set_prev(Prev& p, const Field2& o, float2 r)
{
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        p.E[i] = o.E[i];
        if (!FF) p.B[i] = o.B[i];
    }
    p.S = o.S;
    if (!FF) p.SB = mul2(o.S, o.rinv);
    p.r = r;
}

// running bin of cell j (+)= w times the sample's field
template <bool FF, bool SET>
__device__ __forceinline__ void add_prev(Cells<2>& c, const Prev& p, int j, float w)
{
    const float we = w * half_of(p.S, j), wb = FF ? 0.f : w * half_of(p.SB, j);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        c.acc[i][j] = SET ? half_of(p.E[i], j) * we : fmaf(half_of(p.E[i], j), we, c.acc[i][j]);
        if (!FF) c.acc[3 + i][j] = SET ? half_of(p.B[i], j) * wb : fmaf(half_of(p.B[i], j), wb, c.acc[3 + i][j]);
    }
}

template <bool FF>
__device__ __forceinline__ void add_prev2(Cells<2>& c, const Prev& p, float2 w)
{
    const float2 we = mul2(w, p.S), wb = FF ? w : mul2(w, p.SB);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        c.acc[i][0] = fmaf(p.E[i].x, we.x, c.acc[i][0]);
        c.acc[i][1] = fmaf(p.E[i].y, we.y, c.acc[i][1]);
        if (!FF) {
            c.acc[3 + i][0] = fmaf(p.B[i].x, wb.x, c.acc[3 + i][0]);
            c.acc[3 + i][1] = fmaf(p.B[i].y, wb.y, c.acc[3 + i][1]);
        }
    }
}

// Fast step.  a: the sample whose field this interval completes (k-1; quadratic: k-2),
// b: quadratic: sample k-1; a leaves as sample k (its place in the caller's rotation), b with its new r.
// half_ramp: 1/2, or 0 to hold the previous field; curv: quadratic: 1, or 0 while fewer than three fields
// lie behind.
template <int NT, bool FF, bool QUAD, int TRACK>
__device__ __forceinline__ void lin_step(Cells<2>& c, Prev& a, Prev& b, float2& h, const RecS& r, const Consts& C,
                                         float half_ramp, float curv, const Cold<2, NT>& cold, const Place& at)
{
    Prev n;
    float2 t, iL, al, be;
    {
        Field2 o;
        field_pair<FF>(r, c, C, o);
        t = fma2(o.num, o.rden, pair_of(c.f));
        set_prev<FF>(n, o, both(0.f));
    }
    const float2 f = pair_of(c.f);
    const float2 len1 = sub2(make_float2(fminf(t.x, C.W), fminf(t.y, C.W)), f), L = sub2(t, f);
    iL = make_float2(fast_rcp(fmaxf(L.x, 1e-30f)), fast_rcp(fmaxf(L.y, 1e-30f)));
    const float2 ramp1 = mul2(mul2(both(half_ramp), len1), mul2(len1, iL));
    float2 wp, cu1;                 // weights of the first part: of sample k-1 (wp), of this sample (n.r)
    if (QUAD) {
        const float2 iLh = mul2(both(curv), rcp2(add2(L, h)));
        al = mul2(iL, iLh);
        be = mul2(rcp2(h), iLh);
        cu1 = qcube2(len1, L);
        add_prev2<FF>(c, a, fma2(cu1, be, a.r));
        wp = add2(b.r, sub2(sub2(len1, ramp1), mul2(cu1, add2(al, be))));
        n.r = fma2(cu1, al, ramp1);
    } else {
        add_prev2<FF>(c, a, add2(a.r, sub2(len1, ramp1)));
        n.r = ramp1;
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        float fn = half_of(t, j);
        fn = fn < 2.f * C.W ? fn : -INFINITY;
        c.f[j] = fn;
        if (fn >= C.W) {
            if (QUAD) add_prev<FF, false>(c, b, j, half_of(wp, j));
            add_prev<FF, false>(c, n, j, half_of(n.r, j));
            red_bin<NT, FF, TRACK>(C, c, j, cold, at, at.k);
            const float rem = fn - C.W, Lj = half_of(L, j);
            const float ramp2 = fmaf(half_ramp, Lj, -half_of(ramp1, j));
            if (QUAD) {
                const float cu2 = qcube(Lj, Lj) - half_of(cu1, j);
                add_prev<FF, true>(c, a, j, cu2 * half_of(be, j));
                set_half(wp, j, rem - ramp2 - cu2 * (half_of(al, j) + half_of(be, j)));
                set_half(n.r, j, fmaf(cu2, half_of(al, j), ramp2));
            } else {
                add_prev<FF, true>(c, a, j, rem - ramp2);
                set_half(n.r, j, ramp2);
            }
            c.f[j] = rem;
            c.bo[j] += 1;
        }
    }
    a = n;
    if (QUAD) {
        b.r = wp;
        h = L;
    }
}

// Exact step: any number of edges, bins checked against the window, clipped intervals counted.  again: after
// a fast walk that stopped; ok: false from the interval that stopped it onwards.
template <int NT, bool FF, bool QUAD>
__device__ __forceinline__ void lin_exact_step(Cells<2>& c, LinState& l, const RecS& r, const Consts& C,
                                               const Cold<2, NT>& cold, bool last, int k, int k_begin, int k_end,
                                               float half_ramp, bool again, bool* ok)
{
    Field2 o;
    field_pair<FF>(r, c, C, o);
    Prev n;
    set_prev<FF>(n, o, both(0.f));
    const float curv = (QUAD && k >= C.kq) ? 1.f : 0.f;
    float2 rp = both(0.f), Lk;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const float f = c.f[j];
        const float t = last ? fmaf((float)(cold.bo_end(j) - c.bo[j]), C.W, cold.f_end(j))
                             : fmaf(half_of(o.num, j), half_of(o.rden, j), f);
        const float L = t - f, iL = fast_rcp(fmaxf(L, 1e-30f));
        const float iLh = QUAD ? curv * fast_rcp(L + half_of(l.h, j)) : 0.f;
        const float al = QUAD ? iL * iLh : 0.f, be = QUAD ? fast_rcp(half_of(l.h, j)) * iLh : 0.f;
        // weights of the part [s0, s0 + len] of the interval: of samples k-2, k-1 and k
        auto weights = [&](float s0, float len, float& w2, float& w1, float& w0) {
            const float s1 = s0 + len;
            const float ramp = (half_ramp * iL) * (len * (s0 + s1));
            const float cu = QUAD ? qcube(s1, L) - qcube(s0, L) : 0.f;
            w2 = cu * be;
            w1 = (len - ramp) - cu * (al + be);
            w0 = fmaf(cu, al, ramp);
        };
        ok[j] = ok[j] && t < 2.f * C.W;
        const bool go = !(again && ok[j]);
        int m = t >= C.W ? 1 : 0;
        float rem = t - C.W;
        if (t >= 2.f * C.W) {
            m = max(2, (int)fminf(floorf(t * C.invW), 16777216.f));
            rem = fminf(fmaxf(fmaf(-(float)m, C.W, t), 0.f), C.W * 0.99999994f);
        }
        float w2, w1, w0;
        weights(0.f, fminf(t, C.W) - f, w2, w1, w0);
        if (QUAD) {
            add_prev<FF, false>(c, l.p2, j, half_of(l.p2.r, j) + w2);
            w1 += half_of(l.p1.r, j);
        } else {
            add_prev<FF, false>(c, l.p1, j, half_of(l.p1.r, j) + w1);
        }
        if (m > 0) {
            const int b0 = c.bo[j] - row_base<NT>(j, C.n_bins);
            if (QUAD) add_prev<FF, false>(c, l.p1, j, w1);
            add_prev<FF, false>(c, n, j, w0);
            if (go) flush_acc<2, FF>(C, c, j, b0, c.bo[j]);
            // whole bins b0 + i
            const int hi = go ? min(m - 1, C.n_bins - 1 - b0) : 0;
            for (int i = max(1, -b0); i <= hi; ++i) {
                weights(fmaf((float)i, C.W, -f), C.W, w2, w1, w0);
                add_prev<FF, true>(c, n, j, w0);
                add_prev<FF, false>(c, l.p1, j, w1);
                if (QUAD) add_prev<FF, false>(c, l.p2, j, w2);
                flush_acc<2, FF>(C, c, j, b0 + i, c.bo[j] + i);
            }
            weights(fmaf((float)m, C.W, -f), rem, w2, w1, w0);
            add_prev<FF, true>(c, QUAD ? l.p2 : l.p1, j, QUAD ? w2 : w1);
            c.bo[j] += m;
            if (b0 < 0 && b0 + m >= 0) cold.set(j, kBelow, k - k_begin + 1);
            if (b0 < C.n_bins && b0 + m >= C.n_bins) cold.set(j, kAbove, k_end - k + 1);
        }
        c.f[j] = m > 0 ? rem : t;
        set_half(n.r, j, w0);
        set_half(rp, j, w1);
        set_half(Lk, j, L);
    }
    if (QUAD) {
        l.p2 = l.p1;
        l.p2.r = rp;
        l.h = Lk;
    }
    l.p1 = n;
}

// The weights still to come of the earlier samples' fields, into the running bin (at the chunk's end).
template <bool FF, bool QUAD>
__device__ __forceinline__ void settle(Cells<2>& c, const LinState& l)
{
    add_prev2<FF>(c, l.p1, l.p1.r);
    if (QUAD) add_prev2<FF>(c, l.p2, l.p2.r);
}

// Scratch of a warp in shared memory: save_cell words for each of its 32 NC cells.  The fast walk keeps
// the state at the start of a tile there ([word][lane]: f, rpd, bo, below, above, acc[6]; interpolated
// fields: p1, and for the quadratic interpolation p2 and h); the exact walk, once it has taken that state
// back, hands its runs of finished bins over there (add_runs: 16 words per lane).
constexpr int save_cell(int lin) { return lin == 2 ? 30 : lin == 1 ? 20 : 17; }

template <int NC, int NT, bool TRACK, bool FF>
__device__ __forceinline__ void save_state(const Cells<NC>& c, const Cold<NC, NT>& cold, float (*sv)[32], int words)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < NC; ++j, sv += words) {
        sv[0][lane] = c.f[j];
        sv[1][lane] = c.rpd[j];
        sv[2][lane] = __int_as_float(c.bo[j]);
        if (TRACK) {
            sv[3][lane] = __int_as_float(cold.below(j));
            sv[4][lane] = __int_as_float(cold.above(j));
        }
#pragma unroll
        for (int i = 0; i < (FF ? 3 : 6); ++i) sv[5 + i][lane] = c.acc[i][j];
    }
}

template <int NC, int NT, bool TRACK, bool FF>
__device__ __forceinline__ void restore_state(Cells<NC>& c, const Cold<NC, NT>& cold, const float (*sv)[32], int words)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < NC; ++j, sv += words) {
        c.f[j] = sv[0][lane];
        c.rpd[j] = sv[1][lane];
        c.bo[j] = __float_as_int(sv[2][lane]);
        if (TRACK) {
            cold.set(j, kBelow, sv[3][lane]);
            cold.set(j, kAbove, sv[4][lane]);
        }
#pragma unroll
        for (int i = 0; i < (FF ? 3 : 6); ++i) c.acc[i][j] = sv[5 + i][lane];
    }
}

template <bool FF>
__device__ __forceinline__ void save_prev(const Prev& p, float (*sv)[32], int words)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < 2; ++j, sv += words) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            sv[i][lane] = half_of(p.E[i], j);
            if (!FF) sv[3 + i][lane] = half_of(p.B[i], j);
        }
        sv[6][lane] = half_of(p.S, j);
        if (!FF) sv[7][lane] = half_of(p.SB, j);
        sv[8][lane] = half_of(p.r, j);
    }
}

template <bool FF>
__device__ __forceinline__ void restore_prev(Prev& p, const float (*sv)[32], int words)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < 2; ++j, sv += words) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            set_half(p.E[i], j, sv[i][lane]);
            if (!FF) set_half(p.B[i], j, sv[3 + i][lane]);
        }
        set_half(p.S, j, sv[6][lane]);
        if (!FF) set_half(p.SB, j, sv[7][lane]);
        set_half(p.r, j, sv[8][lane]);
    }
}

// ---------------------------------------------------------------------------------------------
// Exact walk of the held field: any number of bin edges per interval.
//
// Where intervals pass several edges the walk is bound by the reductions: with a lane per cell every
// finished bin is two reductions that share a 128-byte line with no other lane's, which L2 takes at
// 9.2e10 bins/s (5e10 where the detector does not fit it).  Eight lanes adding four consecutive bins of
// one cell with one instruction reach 1.5e11 (8e10; reductions alone, measured).  So where a cell of the
// warp finishes kRunBins bins or more in a step, every lane hands its run over through shared memory and
// groups of eight lanes add the runs.  Measured, deposit kernel, with the exact walk taken at once where
// the tile before needed it (before: fast walk, then exact walk lane by lane): one electron, 38000 steps
// x 512 cells x 131072 bins (3.4 edges a step) 2.17 -> 1.12 ms; 400 steps x 4096 cells x 8192 bins (20 a
// step) 0.322 -> 0.261 ms; 256 electrons x 1200 cells, 25 steps a call (2 a step) 0.195 -> 0.196 ms.
// Gathering whole 128-byte lines of four bins per cell before adding them cost more instructions than
// the fuller lines saved (1.09, 0.338, 0.226 ms).
// ---------------------------------------------------------------------------------------------
// Shortest run, of any cell of the warp, that is handed over; 2, 4 and 6 on the cases above: 0.98, 1.21 and
// 1.61 ms; 0.260, 0.264 and 0.262 ms; 0.216, 0.205 and 0.212 ms.
constexpr int kRunBins = 3;
// Lanes with such a run that make the warp hand them over: the hand-over costs every lane, so a few do better
// alone.  1, 4, 6 and 8 lanes: 680 electrons x 496 steps x 925 cells x 2146 bins (1.5 edges a step) 5.75, 4.98,
// 4.45 and 4.58 ms; the streamed case above 2.85, 2.99, 3.13 and 3.28 ms for its 16 launches.
constexpr int kRunLanes = 6;
// Lane's run: `count` consecutive bins from bin b of cell row j's detector row; bin 0 is `e0`, `h0` (E and
// B) if `first`, every other one `e1`, `h1`.  Called by the converged warp; stage: 32 x 4 float4 of the warp.
template <int NT>
__device__ __forceinline__ void add_runs(const Consts& C, float4* stage, int j, int b, int count, bool first,
                                         const float* e0, const float* h0, const float* e1, const float* h1)
{
    const int lane = threadIdx.x & 31;
    // chunk c of a lane, XORed so that eight lanes' 16-byte stores fall on distinct banks
    auto chunk = [&](int l, int c) -> float4& { return stage[l * 4 + (c ^ ((l >> 1) & 3))]; };
    __syncwarp();
    chunk(lane, 0) = make_float4(e0[0], e0[1], e0[2], h0[0]);
    chunk(lane, 1) = make_float4(h0[1], h0[2], 0.f, 0.f);
    chunk(lane, 2) = make_float4(e1[0], e1[1], e1[2], h1[0]);
    chunk(lane, 3) = make_float4(h1[1], h1[2], 0.f, 0.f);
    __syncwarp();
    const int group = lane >> 3, sub = (lane >> 1) & 3, half = lane & 1;
    const int info = count * 2 + (first ? 1 : 0);
    const int row0 = (j * NT + (int)(threadIdx.x & ~31u) + group) * C.n_bins + sub;
    for (int i0 = 0; __any_sync(0xffffffffu, i0 < count); i0 += 4) {
        const int i = i0 + sub;
#pragma unroll 4
        for (int g = 0; g < 8; ++g) {
            const int owner = 4 * g + group;
            const int ob = __shfl_sync(0xffffffffu, b, owner), oi = __shfl_sync(0xffffffffu, info, owner);
            if (2 * i < (oi & ~1)) {
                const float4 v = chunk(owner, (i == 0 && (oi & 1) ? 0 : 2) + half);
                red_add_v4(bin_addr(C, row0 + 4 * g * C.n_bins + ob + i0) + 4 * half, v.x, v.y, v.z, v.w);
            }
        }
    }
}

template <int NC, int NT, bool FF>
__device__ __forceinline__ bool exact_tile(Cells<NC>& c, const RecS* tile, int cnt, bool last_tile, const Consts& C,
                                           const Cold<NC, NT>& cold, int k0, int k_begin, int k_end, float* scratch,
                                           bool again, bool track)
{
    bool ok[NC];                    // no interval of two or more edges so far
#pragma unroll
    for (int j = 0; j < NC; ++j) ok[j] = true;
#pragma unroll 1
    for (int i = 0; i < cnt; ++i) {
        const RecS& r = tile[i];
        const bool last = last_tile && i == cnt - 1;
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            Field o;
            if (FF)
                field_at_ff(r, c.px[j], c.py[j], c.pz[j], c.rpd[j], c.nlx[j], c.nly[j], c.nlz[j], o);
            else
                field_at(r, c.px[j], c.py[j], c.pz[j], c.rpd[j], C, o);
            const float t = last ? fmaf((float)(cold.bo_end(j) - c.bo[j]), C.W, cold.f_end(j))
                                 : fmaf(o.num, o.rden, c.f[j]);
            const float ws = (fminf(t, C.W) - c.f[j]) * o.S, wb = FF ? ws : ws * o.rinv;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                c.acc[q][j] = fmaf(o.E[q], ws, c.acc[q][j]);
                if (!FF) c.acc[3 + q][j] = fmaf(o.B[q], wb, c.acc[3 + q][j]);
            }
            // edges passed, and the time left in the last bin
            ok[j] = ok[j] && t < 2.f * C.W;
            int m = t >= C.W ? 1 : 0;
            float rem = t - C.W;
            if (t >= 2.f * C.W) {
                // at least two, also where t is 2 W to the last digit and t / W rounds below 2
                m = max(2, (int)fminf(floorf(t * C.invW), 16777216.f));
                // (two roundings: where an edge is met to the last digit, another one would tell it apart)
                rem = fminf(fmaxf(fmaf(-(float)(m - 1), C.W, t), C.W), C.W * 1.99999988f) - C.W;
            }
            // finished bins b0 .. b0 + m - 1, those inside the window: the first from the accumulator, the
            // others whole bins of this interval's field
            const int b0 = c.bo[j] - row_base<NT>(j, C.n_bins);
            const int b = max(b0, 0);
            const int count = again && ok[j] ? 0 : max(0, min(b0 + m, C.n_bins) - b);
            if (__any_sync(0xffffffffu, count > 0)) {
                const bool first = b == b0;         // false: the window starts inside the interval
                const int rest = count - (first ? 1 : 0);
                const float e0[3] = {c.acc[0][j], c.acc[1][j], c.acc[2][j]};
                const float cb[3] = {c.acc[3][j], c.acc[4][j], c.acc[5][j]};
                float h0[3], e1[3], h1[3];
                bin_b<NC, FF>(c, j, e0, cb, h0);
                const bool runs = __popc(__ballot_sync(0xffffffffu, count >= kRunBins)) >= kRunLanes;
                if (!runs && first && count > 0) {
                    float* a = bin_addr(C, c.bo[j]);
                    red_add_v4(a, e0[0], e0[1], e0[2], h0[0]);
                    red_add_v2(a + 4, h0[1], h0[2]);
                }
                if (__any_sync(0xffffffffu, rest > 0)) {
                    const float fs = C.W * o.S, fb = FF ? fs : fs * o.rinv;
                    float cb1[3];
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        e1[q] = o.E[q] * fs;
                        cb1[q] = FF ? 0.f : o.B[q] * fb;
                    }
                    bin_b<NC, FF>(c, j, e1, cb1, h1);
                    if (runs) {
                        add_runs<NT>(C, reinterpret_cast<float4*>(scratch), j, b, count, first, e0, h0, e1, h1);
                    } else {
                        float* a = bin_addr(C, row_base<NT>(j, C.n_bins) + b + (first ? 1 : 0));
#pragma unroll 1
                        for (int q = 0; q < rest; ++q, a += 8) {
                            red_add_v4(a, e1[0], e1[1], e1[2], h1[0]);
                            red_add_v2(a + 4, h1[1], h1[2]);
                        }
                    }
                }
            }
            if (m > 0) {
                const float rs = rem * o.S, rb = FF ? rs : rs * o.rinv;
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    c.acc[q][j] = o.E[q] * rs;
                    if (!FF) c.acc[3 + q][j] = o.B[q] * rb;
                }
                if (track) {
                    if (b0 < 0 && b0 + m >= 0) cold.set(j, kBelow, k0 + i - k_begin + 1);
                    if (b0 < C.n_bins && b0 + m >= C.n_bins) cold.set(j, kAbove, k_end - (k0 + i) + 1);
                }
            }
            c.f[j] = m > 0 ? rem : t;
            c.bo[j] += m;
        }
    }
    bool met = false;
#pragma unroll
    for (int j = 0; j < NC; ++j) met = met || !ok[j];
    __syncwarp();                   // the scratch may hold saved states again
    return __any_sync(0xffffffffu, met);
}

// The fast walk of one tile; false if it met an interval of two or more edges (the state is then back at the
// tile's start).
template <int NC, int NT, int TRACK, bool FF, int LIN>
__device__ __forceinline__ bool fast_tile(Cells<NC>& c, LinState& l, const RecS* tile, int cnt, bool last_tile,
                                          const Consts& C, float half_ramp, const Cold<NC, NT>& cold, int k0, int k_begin,
                                          int k_end, float* scratch, bool track)
{
    constexpr bool QUAD = LIN == 2;
    constexpr int words = save_cell(LIN);
    float (*sv)[32] = reinterpret_cast<float (*)[32]>(scratch);
    const int n_regular = last_tile ? cnt - 1 : cnt;
    save_state<NC, NT, TRACK != kUntracked, FF>(c, cold, sv, words);
    if constexpr (LIN != 0) {
        save_prev<FF>(l.p1, sv + 11, words);
        if (QUAD) {
            const int lane = threadIdx.x & 31;
            save_prev<FF>(l.p2, sv + 20, words);
            sv[29][lane] = l.h.x;
            sv[words + 29][lane] = l.h.y;
        }
        int i = 0;
        if constexpr (QUAD) {
            auto curv = [&](int q) { return k0 + q >= C.kq ? 1.f : 0.f; };
#pragma unroll 1
            for (; i + 1 < n_regular; i += 2) {
                lin_step<NT, FF, true, TRACK>(c, l.p2, l.p1, l.h, tile[i], C, half_ramp, curv(i), cold,
                                              {k0 + i, k_begin, k_end, track});
                lin_step<NT, FF, true, TRACK>(c, l.p1, l.p2, l.h, tile[i + 1], C, half_ramp, curv(i + 1), cold,
                                              {k0 + i + 1, k_begin, k_end, track});
            }
            if (i < n_regular) {
                lin_step<NT, FF, true, TRACK>(c, l.p2, l.p1, l.h, tile[i], C, half_ramp, curv(i), cold,
                                              {k0 + i, k_begin, k_end, track});
                const Prev x = l.p1;
                l.p1 = l.p2;
                l.p2 = x;
            }
        } else {
            // (two per iteration, so that sample k's field stays where it was formed)
#pragma unroll 2
            for (; i < n_regular; ++i)
                lin_step<NT, FF, false, TRACK>(c, l.p1, l.p2, l.h, tile[i], C, half_ramp, 0.f, cold,
                                               {k0 + i, k_begin, k_end, track});
        }
    } else if constexpr (NC == 2) {
        int i = 0;
#pragma unroll 1
        for (; i + 1 < n_regular; i += 2)
            two_steps_pair<NT, FF, TRACK>(c, tile[i], tile[i + 1], C, cold, {k0 + i, k_begin, k_end, track});
        if (i < n_regular) step<NC, NT, false, TRACK != kUntracked, FF>(c, tile[i], C, cold, k0 + i, k_begin, k_end);
    } else {
#pragma unroll kUnroll
        for (int i = 0; i < n_regular; ++i)
            step<NC, NT, false, TRACK != kUntracked, FF>(c, tile[i], C, cold, k0 + i, k_begin, k_end);
    }
    if constexpr (LIN == 0) {
        if (last_tile) step<NC, NT, true, TRACK != kUntracked, FF>(c, tile[cnt - 1], C, cold, k_end, k_begin, k_end);
    }
    bool stopped = false;
#pragma unroll
    for (int j = 0; j < NC; ++j) stopped = stopped || c.f[j] == -INFINITY;
    if (!__any_sync(0xffffffffu, stopped)) {
        if constexpr (LIN != 0) {
            bool ok[2] = {true, true};
            if (last_tile)
                lin_exact_step<NT, FF, QUAD>(c, l, tile[cnt - 1], C, cold, true, k_end, k_begin, k_end, half_ramp, false,
                                             ok);
        }
        return true;
    }
    restore_state<NC, NT, TRACK != kUntracked, FF>(c, cold, sv, words);
    if constexpr (LIN != 0) {
        restore_prev<FF>(l.p1, sv + 11, words);
        if (QUAD) {
            const int lane = threadIdx.x & 31;
            restore_prev<FF>(l.p2, sv + 20, words);
            l.h = make_float2(sv[29][lane], sv[words + 29][lane]);
        }
    }
    return false;
}

// The exact walk of one tile; again: after a fast walk that stopped (earlier bins are flushed).  Returns
// whether the warp met an interval of two or more edges.
template <int NC, int NT, bool FF, int LIN>
__device__ __forceinline__ bool exact_walk(Cells<NC>& c, LinState& l, const RecS* tile, int cnt, bool last_tile,
                                           const Consts& C, float half_ramp, const Cold<NC, NT>& cold, int k0, int k_begin,
                                           int k_end, float* scratch, bool again, bool track)
{
    if constexpr (LIN == 0) {
        return exact_tile<NC, NT, FF>(c, tile, cnt, last_tile, C, cold, k0, k_begin, k_end, scratch, again, track);
    } else {
        bool ok[2] = {true, true};
#pragma unroll 1
        for (int i = 0; i < cnt; ++i) {
            const bool last = last_tile && i == cnt - 1;        // (not walked by a fast walk that stopped)
            lin_exact_step<NT, FF, LIN == 2>(c, l, tile[i], C, cold, last, k0 + i, k_begin, k_end, half_ramp,
                                             again && !last, ok);
        }
        return __any_sync(0xffffffffu, !ok[0] || !ok[1]);
    }
}

// The walk of a chunk's tiles, the first two of which are being copied; false if a bounded wait ran out (the error
// is recorded).  track: some bin of the CTA's walk may lie outside the window.  The tracked fast walk costs a few
// instructions where an edge is passed, but beside the untracked one it also costs that one registers, differently in
// each kernel, so each has the form that measured best.  TRACK says which: kUntracked or kTracked, a loop over the
// tiles for each (held field); kTrackFlag, one loop, with a fast walk for each or, for the quadratic interpolation,
// one walk that reads the flag.  Measured (ms, whole window; window without a quarter of the arrivals at each end), 100
// electrons x 1500 steps x 10000 cells x 1500 bins, interpolated chunks at a window's end all in the exact walk: held
// 5.45; 5.50, linear 5.63; 7.82, quadratic 7.34; 10.12; a loop for each: held 5.35; 5.16, linear 5.75; 6.01, quadratic
// 7.64; 7.83; a walk for each: held 5.44; 5.25, linear 5.65; 5.78, quadratic 7.55; 8.28; by the flag: linear 5.83; 6.12,
// quadratic 7.43; 7.93.  (The tracked walk as a call, out of line: held 5.41; 5.60, linear 5.76; 6.80.)
template <int NC, int NT, int TRACK, bool FF, int LIN>
__device__ __forceinline__ bool walk_tiles(const DepositParams& P, Cells<NC>& c, LinState& l, const Consts& C,
                                           const Cold<NC, NT>& cold, const RecS* rec, RecS (*tile)[kTileSteps], uint64_t* bar,
                                           unsigned g_base, int n_tiles, int k_begin, int k_end, bool many, bool track,
                                           float* scratch)
{
    const int tid = threadIdx.x;
    for (int t = 0; t < n_tiles; ++t) {
        const unsigned g = g_base + t;
        const int buf = g & 1;
        const bool ok = mbar_wait_bounded(&bar[buf], (g >> 1) & 1u);
        if (__syncthreads_or(!ok)) {
            // a bulk copy did not complete: record it, let outstanding copies land, stop.
            if (tid == 0) {
                atomicOr(&P.counters->errors, ERRBIT_TIMEOUT);
                for (int u = t; u < t + 2 && u < n_tiles; ++u)
                    (void)mbar_wait_bounded(&bar[(g_base + u) & 1], ((g_base + u) >> 1) & 1u);
            }
            __syncthreads();
            return false;
        }
        const int k0 = k_begin + t * kTileSteps;
        const int cnt = min(kTileSteps, k_end - k0 + 1);
        const bool last_tile = (t == n_tiles - 1);
        // many (warp-uniform): the warp's last tile met intervals of two or more edges (at the start: the
        // anchors say more than one edge an interval), so this one goes to the exact walk at once
        const float half_ramp = P.lin == 2 ? 0.f : 0.5f;
        bool done = false;
        if (!many) {
            if constexpr (TRACK == kTrackFlag && LIN != 2)
                done = track ? fast_tile<NC, NT, kTracked, FF, LIN>(c, l, tile[buf], cnt, last_tile, C, half_ramp, cold, k0,
                                                                    k_begin, k_end, scratch, true)
                             : fast_tile<NC, NT, kUntracked, FF, LIN>(c, l, tile[buf], cnt, last_tile, C, half_ramp, cold, k0,
                                                                      k_begin, k_end, scratch, false);
            else
                done = fast_tile<NC, NT, TRACK, FF, LIN>(c, l, tile[buf], cnt, last_tile, C, half_ramp, cold, k0, k_begin,
                                                         k_end, scratch, track);
        }
        if (!done)
            many = exact_walk<NC, NT, FF, LIN>(c, l, tile[buf], cnt, last_tile, C, half_ramp, cold, k0, k_begin, k_end,
                                               scratch, !many, track);
        __syncthreads();
        if (tid == 0 && t + 2 < n_tiles) {
            fence_proxy_async();
            const int k2 = k_begin + (t + 2) * kTileSteps;
            const unsigned bytes = (unsigned)min(kTileSteps, k_end - k2 + 1) * sizeof(RecS);
            mbar_arrive_expect_tx(&bar[buf], bytes);
            bulk_g2s(tile[buf], rec + k2, bytes, &bar[buf]);
        }
    }
    return true;
}

}  // namespace

// One work item -- particle p, cell block cb, step chunk ch of one problem -- run by the whole
// CTA.  tile / bar: the CTA's shared staging buffers; g_base counts the tiles the CTA staged
// before this item (it selects buffer and mbarrier phase, so the buffers carry over between items).
// Returns false if a bounded wait ran out (the error is recorded; the CTA must stop).
template <bool FF, int LIN, int NC, int CPC>
__device__ __forceinline__ bool deposit_item(const DepositParams& P, int p, int cb, int ch,
                                             RecS (*tile)[kTileSteps], uint64_t* bar, float (*cold_words)[CPC / NC],
                                             float* scratch, unsigned& g_base)
{
    constexpr int NT = CPC / NC;                // threads of the CTA
    const int S = P.n_samples - 1;
    const int k_begin = P.k_first + ch * P.chunk;
    const int k_end = min(S, k_begin + P.chunk - 1);
    const int n_int = k_end - k_begin + 1;
    const int n_tiles = (n_int + kTileSteps - 1) / kTileSteps;
    const RecS* rec = static_cast<const RecS*>(P.rec) + (size_t)p * P.n_samples;
    const int tid = threadIdx.x;

    if (tid == 0) {
        fence_proxy_async();
        for (int t = 0; t < 2 && t < n_tiles; ++t) {
            const int k0 = k_begin + t * kTileSteps;
            const unsigned g = g_base + t;
            const unsigned bytes = (unsigned)min(kTileSteps, k_end - k0 + 1) * sizeof(RecS);
            mbar_arrive_expect_tx(&bar[g & 1], bytes);
            bulk_g2s(tile[g & 1], rec + k0, bytes, &bar[g & 1]);
        }
    }

    Consts C;
    C.W = P.W;
    C.invW = P.invW;
    C.DT = P.dt_f;
    C.n_bins = P.n_bins;
    C.base = static_cast<float*>(P.fields) + (size_t)cb * CPC * P.n_bins * 8;
    C.kq = 3 - P.k_real0;
#if RD_CHECK
    C.errors = &P.counters->errors;
#endif
    constexpr bool QUAD = LIN == 2;
    const bool q_prev = QUAD && k_begin >= 3;     // the chunk starts with three fields behind it

    // anchors: exact FP64 arrival (bins) at both ends of the chunk, per cell
    Cells<NC> c;
    const Cold<NC, NT> cold{cold_words};
    scratch += (tid >> 5) * 32 * NC * save_cell(LIN);       // this warp's part
    float hp0[NC];                              // quadratic: length of interval k_begin - 1 (dt units)
    bool partial = false, many = false;
    unsigned long long clip = 0, crossed = 0;
    const double* xp = P.x + (size_t)p * P.n_samples * 3;
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        const int row = j * NT + tid;
        const int cell = cb * CPC + row;
        // a cell without arrivals in the window still walks (no per-cell branch in the step) but
        // from a time that never reaches a bin edge: nothing is flushed
        const int rb = row * P.n_bins;
        c.bo[j] = rb;
        c.f[j] = -1e30f;
        c.rpd[j] = 1e6f;
        c.px[j] = 1e6f;
        c.py[j] = c.pz[j] = 0.f;
        c.nlx[j] = c.nly[j] = c.nlz[j] = 0.f;
        int bo_end = rb, below = -1;
        hp0[j] = 1.f;
        float f_end = 0.f;
#pragma unroll
        for (int i = 0; i < 6; ++i) c.acc[i][j] = 0.f;
        if (cell < P.n_pix) {
            const D4 cl = P.cells[cell];
            const double* xa = xp + 3 * (size_t)(k_begin - 1);
            const double* xe = xp + 3 * (size_t)k_end;
            double Ra = 0.0, Re, ua, ue, ncx = 0.0, ncy = 0.0, ncz = 0.0, Rc = 1.0;
            if (FF) {
                farfield_cell(cl, ncx, ncy, ncz, Rc);
                ua = arrival_bins_ff(xa[0], xa[1], xa[2], ncx, ncy, ncz, Rc, cl.w, P.t0, k_begin - 1, P.dt, P.inv_dt_det);
                ue = arrival_bins_ff(xe[0], xe[1], xe[2], ncx, ncy, ncz, Rc, cl.w, P.t0, k_end, P.dt, P.inv_dt_det);
            } else {
                ua = arrival_bins(xa[0], xa[1], xa[2], cl, P.t0, k_begin - 1, P.dt, P.inv_dt_det, Ra);
                ue = arrival_bins(xe[0], xe[1], xe[2], cl, P.t0, k_end, P.dt, P.inv_dt_det, Re);
            }
            const bool live = (ue > 0.0) && (ua < (double)P.n_bins);
            if (q_prev && live) {
                const double* xq = xp + 3 * (size_t)(k_begin - 2);
                double Rq;
                const double uq =
                    FF ? arrival_bins_ff(xq[0], xq[1], xq[2], ncx, ncy, ncz, Rc, cl.w, P.t0, k_begin - 2, P.dt,
                                         P.inv_dt_det)
                       : arrival_bins(xq[0], xq[1], xq[2], cl, P.t0, k_begin - 2, P.dt, P.inv_dt_det, Rq);
                hp0[j] = (float)((ua - uq) * P.W);
            }
            if (!live) {
                clip += (unsigned long long)n_int;
            } else {
                const double fla = floor(ua), fle = floor(ue);
                c.bo[j] = rb + walk_bin(fla);
                c.f[j] = (float)(ua - fla) * P.W;
                bo_end = rb + walk_bin(fle);
                f_end = (float)(ue - fle) * P.W;
                if (FF) {
                    c.px[j] = (float)ncx;
                    c.py[j] = (float)ncy;
                    c.pz[j] = (float)ncz;
                    c.rpd[j] = (float)(1.0 / Rc);
                    c.nlx[j] = (float)(ncx - (double)c.px[j]);
                    c.nly[j] = (float)(ncy - (double)c.py[j]);
                    c.nlz[j] = (float)(ncz - (double)c.pz[j]);
                } else {
                    c.rpd[j] = (float)Ra + P.dt_f;
                    c.px[j] = (float)cl.x;
                    c.py[j] = (float)cl.y;
                    c.pz[j] = (float)cl.z;
                }
                below = (ua < 0.0) ? n_int : 0;
                // unchecked bins need a margin of one bin to each window edge (the FP32 walk may
                // drift by far less than a bin before the end anchor corrects it)
                partial = partial || (ua < 1.0) || (ue > (double)P.n_bins - 1.0);
                crossed += (unsigned long long)max(0, bo_end - c.bo[j]);
                many = many || bo_end - c.bo[j] > n_int;
            }
        }
        cold.set(j, kBoEnd, bo_end);
        cold.set(j, kFEnd, f_end);
        cold.set(j, kBelow, below);
        cold.set(j, kAbove, 0);
    }
    if (clip) atomicAdd(&P.counters->clipped, clip);
    // warp-aggregated count of bin edges crossed (bins touched = intervals + crossings)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) crossed += __shfl_xor_sync(0xffffffffu, crossed, o);
    if ((tid & 31) == 0 && crossed) atomicAdd(&P.counters->crossings, crossed);
    LinState l;
    if constexpr (LIN != 0) {
        // field of the sample before the chunk; a trajectory's first interval holds F_1 (sample 0
        // has no field), so the first chunk starts from the field of sample 1 itself
        const float rpd[2] = {c.rpd[0], c.rpd[1]};
        Field2 o;
        field_pair<FF>(rec[k_begin > 1 ? k_begin - 1 : 1], c, C, o);
        set_prev<FF>(l.p1, o, both(0.f));
        if (QUAD) {
            // the field two samples before the chunk and the interval before it (used from the
            // trajectory's third interval on)
            l.h = make_float2(hp0[0], hp0[1]);
            if (q_prev) field_pair<FF>(rec[k_begin - 2], c, C, o);
            set_prev<FF>(l.p2, o, both(0.f));
        }
        set_pair(c.rpd, pair_of(rpd));
    }
    // clip tracking costs instructions in the bin-crossing path: only CTAs that need it use it
    const bool track = __syncthreads_or(partial) != 0;
    many = __any_sync(0xffffffffu, many);

    bool done;
    if constexpr (LIN == 0 && !FF)
        done = track ? walk_tiles<NC, NT, kTracked, FF, LIN>(P, c, l, C, cold, rec, tile, bar, g_base, n_tiles, k_begin, k_end,
                                                             many, true, scratch)
                     : walk_tiles<NC, NT, kUntracked, FF, LIN>(P, c, l, C, cold, rec, tile, bar, g_base, n_tiles, k_begin,
                                                               k_end, many, false, scratch);
    else
        done = walk_tiles<NC, NT, kTrackFlag, FF, LIN>(P, c, l, C, cold, rec, tile, bar, g_base, n_tiles, k_begin, k_end, many,
                                                       track, scratch);
    if (!done) return false;
    g_base += (unsigned)n_tiles;
    if constexpr (LIN != 0) settle<FF, QUAD>(c, l);
    // close the last bin; count clipped intervals
    unsigned long long clipped = 0;
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        const int below = cold.below(j);
        if (below >= 0) {
            flush_acc<NC, FF>(C, c, j, c.bo[j] - row_base<NT>(j, P.n_bins), c.bo[j]);
            clipped += (unsigned long long)min(n_int, below + cold.above(j));
        }
    }
    if (clipped) atomicAdd(&P.counters->clipped, clipped);
    return true;
}

__device__ __forceinline__ void init_staging(uint64_t* bar)
{
    if (threadIdx.x == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
    }
    __syncthreads();
}

// Resident CTAs per SM the register allotment must allow.  The default CTA (128 threads): 4 for the held
// field's paired walk and the interpolated walks (their state needs 110-128 registers), 5 for the far field's
// held walk.  Other CTA sizes: 512 threads per SM where two cells per thread take the paired walk, as in the
// default shape (128 x 2 and 64 x 2, 37 electrons x 3001 steps x 3233 cells: 1.01 and 1.02 ms at 640 threads, 0.90 and
// 0.90 at 512; 100 x 1500 x 10000 cells: 5.57 and 5.82, 5.45 and 5.69), 640 with one.
#ifndef RD_QUAD_MINBLOCKS
#define RD_QUAD_MINBLOCKS 4
#endif
#ifndef RD_FF_MINBLOCKS
#define RD_FF_MINBLOCKS 5
#endif
#ifndef RD_LIN_MINBLOCKS
#define RD_LIN_MINBLOCKS 4
#endif
constexpr int mixed_min_blocks(int nt, bool ff, int lin, int nc)
{
    if (nt != 128) return (nc == 2 ? 512 : 640) / nt;
    return lin == 2 ? RD_QUAD_MINBLOCKS : lin == 1 ? RD_LIN_MINBLOCKS : ff ? RD_FF_MINBLOCKS : RD_MIXED_MINBLOCKS;
}

template <bool FF, int LIN, int NC, int CPC>
__global__ void __launch_bounds__(CPC / NC, mixed_min_blocks(CPC / NC, FF, LIN, NC)) k_deposit_mixed(const DepositParams P)
{
    constexpr int NT = CPC / NC;
    __shared__ __align__(128) RecS tile[2][kTileSteps];
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ float cold[NC * kColdWords][NT];
    __shared__ __align__(16) float scratch[CPC * save_cell(LIN)];
    init_staging(bar);
    int p, cb, ch;
    item_coords(blockIdx.x, P, p, cb, ch);
    unsigned g = 0;
    (void)deposit_item<FF, LIN, NC, CPC>(P, p, cb, ch, tile, bar, cold, scratch, g);
}

// Persistent form: the resident CTAs draw work items of all problems from one counter.
// Items of problem i are [item_off[i], item_off[i+1]), ordered by item_coords like the
// single-problem grid.  The counter only grows (atomicAdd): no CTA ever waits on another.  One
// instantiation per walk family (far field or not x held / linear family / quadratic): a launch
// holds problems of one family, so the kernel carries only that walk's registers and shared
// state.  (Drawing the next item while walking the current one measured 8 % slower: the drawing
// thread then waits on the atomic before it issues the current item's record copies.)
template <bool FF, int LIN>
__global__ void __launch_bounds__(kMixedThreads, mixed_min_blocks(kMixedThreads, FF, LIN, kMixedCells))
    k_deposit_batch(const DepositParams* __restrict__ probs, const long long* __restrict__ item_off, int n_probs,
                    unsigned long long* next_item)
{
    __shared__ __align__(128) RecS tile[2][kTileSteps];
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ long long s_next;
    __shared__ float cold[kMixedCells * kColdWords][kMixedThreads];
    __shared__ __align__(16) float scratch[kMixedCellsPerCta * save_cell(LIN)];
    init_staging(bar);
    const long long total = item_off[n_probs];
    unsigned g = 0;
    for (;;) {
        if (threadIdx.x == 0) s_next = (long long)atomicAdd(next_item, 1ull);
        __syncthreads();
        const long long item = s_next;
        if (item >= total) break;
        int lo = 0, hi = n_probs - 1;
        while (lo < hi) {                       // last problem whose first item <= item
            const int mid = (lo + hi + 1) >> 1;
            if (item_off[mid] <= item) lo = mid;
            else hi = mid - 1;
        }
        const DepositParams P = probs[lo];
        int p, cb, ch;
        item_coords((unsigned)(item - item_off[lo]), P, p, cb, ch);
        if (!deposit_item<FF, LIN, kMixedCells, kMixedCellsPerCta>(P, p, cb, ch, tile, bar, cold, scratch, g)) break;
    }
}

cudaError_t launch_deposit_batch(int family, const DepositParams* probs, const long long* item_off, int n_probs,
                                 unsigned long long* next_item, cudaStream_t s)
{
    const int grid = batch_grid(family);
    switch (family) {
    case 0: k_deposit_batch<false, 0><<<grid, kMixedThreads, 0, s>>>(probs, item_off, n_probs, next_item); break;
    case 1: k_deposit_batch<false, 1><<<grid, kMixedThreads, 0, s>>>(probs, item_off, n_probs, next_item); break;
    case 2: k_deposit_batch<false, 2><<<grid, kMixedThreads, 0, s>>>(probs, item_off, n_probs, next_item); break;
    case 4: k_deposit_batch<true, 0><<<grid, kMixedThreads, 0, s>>>(probs, item_off, n_probs, next_item); break;
    case 5: k_deposit_batch<true, 1><<<grid, kMixedThreads, 0, s>>>(probs, item_off, n_probs, next_item); break;
    case 6: k_deposit_batch<true, 2><<<grid, kMixedThreads, 0, s>>>(probs, item_off, n_probs, next_item); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <bool FF, int LIN>
static int resident_batch_ctas()
{
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_deposit_batch<FF, LIN>, kMixedThreads, 0);
    return std::max(1, per_sm);
}

int batch_grid(int family)
{
    int per_sm = 1;
    switch (family) {
    case 0: per_sm = resident_batch_ctas<false, 0>(); break;
    case 1: per_sm = resident_batch_ctas<false, 1>(); break;
    case 2: per_sm = resident_batch_ctas<false, 2>(); break;
    case 4: per_sm = resident_batch_ctas<true, 0>(); break;
    case 5: per_sm = resident_batch_ctas<true, 1>(); break;
    case 6: per_sm = resident_batch_ctas<true, 2>(); break;
    default: break;
    }
    return sm_count() * per_sm;
}

#ifndef RD_CARVEOUT
#define RD_CARVEOUT 0
#endif

template <bool FF, int LIN, int NC, int CPC>
static void launch_mixed(const DepositParams& p, unsigned blocks, cudaStream_t s)
{
    if (RD_CARVEOUT) {
        // the largest shared-memory carveout, so that shared memory does not cap the resident CTAs
        static bool done = false;
        if (!done) {
            cudaFuncSetAttribute(k_deposit_mixed<FF, LIN, NC, CPC>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared);
            done = true;
        }
    }
    k_deposit_mixed<FF, LIN, NC, CPC><<<blocks, CPC / NC, 0, s>>>(p);
}

bool mixed_shape_supported(int cells_per_cta, int cells_per_thread)
{
    return (cells_per_cta == 64 || cells_per_cta == 128 || cells_per_cta == 256) &&
           (cells_per_thread == 1 || cells_per_thread == 2);
}

// A grid of the default shape that the multiprocessors hold in one wave waits on latency: one cell per thread and 64
// cells per CTA double the warps and spread them (the results are the same bit for bit but for the order of
// reductions).  For calls whose shape nobody set.  1 x 400 steps x 4096 cells x 8192 bins (128 CTAs): 0.360 -> 0.256
// ms; 1 x 2000 x 64 cells (33): 17.0 -> 16.2 us.
void shape_small_grid(DepositParams& p)
{
    if (p.ff || p.lin || (long long)p.n_cell_blocks * p.n_part * p.n_chunks > 4LL * sm_count()) return;
    p.cpc = 64;
    p.nc = 1;
    p.n_cell_blocks = (p.n_pix + 63) / 64;
    p.group = std::min(p.group * (kMixedCellsPerCta / 64), p.n_cell_blocks);
}

cudaError_t launch_deposit_mixed(const DepositParams& p, cudaStream_t s)
{
    const long long blocks = (long long)p.n_cell_blocks * p.n_part * p.n_chunks;
    if (blocks <= 0) return cudaSuccess;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    const unsigned b = (unsigned)blocks;
    if (p.ff || p.lin) {
        // the far-field and interpolation variants run in the default shape only
        if (p.cpc != kMixedCellsPerCta || p.nc != kMixedCells) return cudaErrorInvalidValue;
        const int lm = p.lin == 3 ? 2 : p.lin ? 1 : 0;       // walk: held, linear family, quadratic
        if (p.ff) {
            if (lm == 2) launch_mixed<true, 2, kMixedCells, kMixedCellsPerCta>(p, b, s);
            else if (lm == 1) launch_mixed<true, 1, kMixedCells, kMixedCellsPerCta>(p, b, s);
            else launch_mixed<true, 0, kMixedCells, kMixedCellsPerCta>(p, b, s);
        } else {
            if (lm == 2) launch_mixed<false, 2, kMixedCells, kMixedCellsPerCta>(p, b, s);
            else launch_mixed<false, 1, kMixedCells, kMixedCellsPerCta>(p, b, s);
        }
        return cudaGetLastError();
    }
    switch (p.cpc * 8 + p.nc) {
    case 256 * 8 + 2: launch_mixed<false, 0, 2, 256>(p, b, s); break;
    case 128 * 8 + 2: launch_mixed<false, 0, 2, 128>(p, b, s); break;
    case 64 * 8 + 2: launch_mixed<false, 0, 2, 64>(p, b, s); break;
    case 256 * 8 + 1: launch_mixed<false, 0, 1, 256>(p, b, s); break;
    case 128 * 8 + 1: launch_mixed<false, 0, 1, 128>(p, b, s); break;
    case 64 * 8 + 1: launch_mixed<false, 0, 1, 64>(p, b, s); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace rd
