// rc_aux.cu -- state set-up, read-out and FP64 diagnostics kernels of the
// RC-LBM library (arXiv 2103.02119, Sec. 4), for sm_103a.
//
// The stored state is post-collision and in pull form (see lbm_device.cuh):
// slot i of cell c is what the next step pulls into cell c + e_i, or, when
// c + e_i is a wall or solid node, what cell c pulls back as direction
// opp(i).  Setting a state scatters distributions into that form; reading it
// gathers them with the same pull the step kernel uses.
#include "lbm_device.cuh"
#include "lbm_launch.h"

namespace lbm {

namespace {

constexpr int kThreads = 256;

// Target cell of direction i from (x, y), wrapped on periodic axes.  Only
// called when the target is a fluid cell (so inside the domain).
__device__ __forceinline__ long long target(const AuxParams& p, int x, int y, int i) {
    int tx = x + ex(i), ty = y + ey(i);
    if (tx < 0) tx += p.nx; else if (tx >= p.nx) tx -= p.nx;
    if (ty < 0) ty += p.ny; else if (ty >= p.ny) ty -= p.ny;
    return (long long)ty * p.nx + tx;
}

// FP32 storage carries the rest part analytically, as the step does: with
// the 1-D factors X = X0 + dX (along x) and Y = Y0 + dY (along y), X0 Y0 =
// w_i,
//   r X Y - rho0 X0 Y0 = (r - rho0) X Y + rho0 (dX Y + X0 dY),
// where dX, dY vanish with the velocity, so FP32 only forms small numbers
// (and GB300's FP64 pipe, a small fraction of its FP32 rate, stays idle).
// The state comes in FP32 too: dr = r - rho0, (u, v).
struct Feq32 {
    float cs2, a, iah2, rho0;
    __device__ __forceinline__ float operator()(int i, float dr, float u, float v) const {
        // The fused multiply-adds are written out: a state that amplifies its
        // last bits (an unstable flow) has to be the same whatever the code
        // around this expression lets the compiler contract.
        const int sx = ex(i), sy = ey(i);
        const float X0 = sx == 0 ? 1.0f - cs2 : 0.5f * cs2;
        const float dX = sx == 0 ? __fmul_rn(-u, u) : 0.5f * __fmaf_rn(u, u, (float)sx * u);
        const float Y0 = sy == 0 ? __fmaf_rn(-2.0f * iah2, cs2, 1.0f) : __fmul_rn(iah2, cs2);
        const float dY = sy == 0 ? __fmul_rn(-2.0f * iah2 * v, v)
                                 : __fmul_rn(iah2, __fmaf_rn(v, v, __fmul_rn((float)sy * a, v)));
        const float X = __fadd_rn(X0, dX), Y = __fadd_rn(Y0, dY);
        const float d = __fmaf_rn(X0, dY, __fmul_rn(dX, Y));
        return __fmaf_rn(__fmul_rn(dr, X), Y, __fmul_rn(rho0, d));
    }
};

// One row per block row of the grid, x across the block: no division of a
// cell index.
#define LBM_FOR_CELLS(p)                                                                 \
    for (int y = blockIdx.y; y < (p).ny; y += gridDim.y)                                 \
        for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < (p).nx;                  \
             x += gridDim.x * blockDim.x)

// Cells c, consecutive over a block and from one row to the next, with their row and
// column: the row by a multiplication with the reciprocal of nx, one of 32 by 32 bits
// below 2^31 cells, else of 64 by 64 with ceil(2^64 / nx), exact while nx times the
// number of cells stays below 2^64 (the latter at every size cost the read-outs of a
// 2048 x 2047 lattice 2 %).  Tiles of one row of 256 columns, or of 2 to 8
// rows of 128 to 32, need no multiplication but leave most threads of a narrow lattice
// without a cell: 3 x 100000, lbm_get_f 62 us against 25, FP64 lbm_diagnostics 435 / 79;
// 2049 x 2048 with obstacles, FP64, 123 / 112 and 578 / 550.
__device__ __forceinline__ int row_of(const AuxParams& p, long long c) {
    if (p.div_shift) return (int)((unsigned long long)(unsigned)c * p.div_mul >> p.div_shift);
    return (int)__umul64hi((unsigned long long)c, p.inv_nx);
}
#define LBM_FOR_ALL_CELLS(p, c)                                                          \
    for (long long c = blockIdx.x * (long long)kThreads + threadIdx.x,                   \
                   n_ = (long long)(p).nx * (p).ny;                                      \
         c < n_; c += gridDim.x * (long long)kThreads)

// GB300 has two FP64 lanes per SM (against 128 FP32 and 64 integer ones): the
// read-out kernels are bound by them, and by conversions, which take the same
// lanes.  So they spend FP64 on what needs it and the rest on integers.
// Measured on 2048 x 2047 FP32 cells with obstacles, against sums, conversions
// and divisions in FP64: lbm_stress 445 against 2010 us (558 with the conversion
// instruction for the sums, 516 with ten FP64 operations more in its algebra),
// lbm_diagnostics after a step 337 against 1153 us (375), lbm_get_f 105 against 145 us,
// lbm_set_f 95 against 146 us, lbm_moments 52 against 69 us; the residual check of a
// 96-lattice batch 0.80 against 2.56 ms (0.86).

// float -> double, exact, on the integer pipe, without a branch (a conversion
// instruction under a predicate takes its place in the FP64 pipe even where
// the predicate is false).
__device__ __forceinline__ double widen(float f) {
    const bool tiny = (__float_as_uint(f) & 0x7F800000u) == 0u;  // subnormal or zero
    const unsigned u = __float_as_uint(tiny ? f * 18446744073709551616.0f : f);  // 2^64
    const unsigned m = u & 0x7FFFFFFFu;
    unsigned hi = (m >> 3) + (tiny ? 0x38000000u - (64u << 20) : 0x38000000u);
    if (m >= 0x7F800000u) hi += 0x38000000u;  // Inf, NaN
    return __hiloint2double((int)((u & 0x80000000u) | (m ? hi : 0u)), (int)(m << 29));
}
__device__ __forceinline__ double widen(double f) { return f; }

// double -> float, rounded to nearest even, on the integer pipe; values that
// are not normal floats below 2^127 (zero aside) through a call.
__device__ __noinline__ float narrow_any(double d) { return (float)d; }
__device__ __forceinline__ float narrow(double d) {
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const unsigned m = hi & 0x7FFFFFFFu;
    unsigned u = ((m - 0x38000000u) << 3) | (lo >> 29);
    const unsigned rest = lo << 3;
    u += (rest > 0x80000000u || (rest == 0x80000000u && (u & 1u))) ? 1u : 0u;
    if (m - 0x38100000u >= 0x47E00000u - 0x38100000u) {
        if (m | lo) return narrow_any(d);
        u = 0u;
    }
    return __uint_as_float((hi & 0x80000000u) | u);
}

// 1 / a for normal a away from the ends of the range: the hardware's
// approximation (about 2^-23) and two Newton steps, four FP64 operations
// (below 1 ulp; an IEEE division takes two to three times as many).
__device__ __forceinline__ double rcp64(double a) {
    double x;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(a));
    x = fma(x, fma(-a, x, 1.0), x);
    return fma(x, fma(-a, x, 1.0), x);
}
__device__ __forceinline__ bool rcp64_ok(double a) {  // 2^-900 <= |a| < 2^900
    const unsigned m = (unsigned)__double2hiint(a) & 0x7FFFFFFFu;
    return m - ((1023u - 900u) << 20) < (1800u << 20);
}

// Sums of the nine deviations of a cell: d = sum g, jx = sum g e_x, jy = sum
// g e_y, sxx = sum g e_x^2, syy, sxy likewise (e_y in units of a).
struct Raw {
    double d, jx, jy, sxx, syy, sxy;
};
template <typename T>
__device__ __forceinline__ Raw raw_sums64(const T g[9]) {
    double w[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) w[i] = widen(g[i]);
    const double se = w[5] + w[8], sw = w[6] + w[7], sm = w[2] + w[4];
    const double ke = w[1] + se, kw = w[3] + sw;
    const double de = w[5] - w[8], dw = w[6] - w[7];
    Raw r;
    r.sxx = ke + kw;
    r.d = (w[0] + sm) + r.sxx;
    r.jx = ke - kw;
    r.jy = (w[2] - w[4]) + (de + dw);
    r.syy = sm + (se + sw);
    r.sxy = de - dw;
    return r;
}

// FP32 storage: the deviations as multiples of 2^-kFixedShift in 64-bit
// integers, where all nine are exact (each zero, or between 2^-35 and 2 in
// magnitude), so that the sums are exact and cost integer instructions.
constexpr int kFixedShift = 58;
__device__ __forceinline__ bool fixed_of(float f, long long& v) {
    const unsigned u = __float_as_uint(f), m = u & 0x7FFFFFFFu;
    const int sh = (int)(m >> 23) - (150 - kFixedShift);
    const unsigned long long a = (unsigned long long)((m & 0x007FFFFFu) | 0x00800000u) << (sh & 63);
    v = (int)u < 0 ? -(long long)a : (long long)a;
    if (m == 0u) v = 0;
    return m == 0u || (sh >= 0 && m < 0x40000000u);
}
// an integer multiple of 2^-kFixedShift as a double (rounded to nearest even),
// on the integer pipe: the conversion instruction takes FP64 lanes
__device__ __forceinline__ double unfixed(long long v) {
    const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const int lz = __clzll((long long)a);
    const unsigned long long n = a << (lz & 63);  // leading bit at 63
    // the 53 leading bits, the hidden one among them: it adds one to the exponent
    unsigned long long m = n >> 11;
    m += ((unsigned)n & 0x7FFu) + ((unsigned)m & 1u) > 0x400u ? 1u : 0u;
    const unsigned e = (unsigned)(1023 + 63 - kFixedShift - 1 - lz) << 20;
    const unsigned hi = ((unsigned)(m >> 32) + e) | ((unsigned)(v >> 32) & 0x80000000u);
    return __hiloint2double(v ? (int)hi : 0, v ? (int)(unsigned)m : 0);
}
// fixed: d in the fixed point (valid when the result is true)
__device__ __forceinline__ bool raw_sums(const float g[9], Raw& r, long long& fixed) {
    long long w[9];
    bool ok = true;
#pragma unroll
    for (int i = 0; i < 9; ++i) ok &= fixed_of(g[i], w[i]);
    fixed = 0;
    if (!ok) {
        r = raw_sums64(g);
        return false;
    }
    const long long se = w[5] + w[8], sw = w[6] + w[7], sm = w[2] + w[4];
    const long long ke = w[1] + se, kw = w[3] + sw;
    const long long de = w[5] - w[8], dw = w[6] - w[7];
    fixed = w[0] + sm + ke + kw;
    r.d = unfixed(fixed);
    r.jx = unfixed(ke - kw);
    r.jy = unfixed(w[2] - w[4] + de + dw);
    r.sxx = unfixed(ke + kw);
    r.syy = unfixed(sm + se + sw);
    r.sxy = unfixed(de - dw);
    return true;
}
__device__ __forceinline__ bool raw_sums(const double g[9], Raw& r, long long& fixed) {
    fixed = 0;
    r = raw_sums64(g);
    return false;
}

// j / rho for both components
__device__ __forceinline__ void over_rho(double rho, double jx, double jy, double& ux,
                                         double& uy) {
    if (rcp64_ok(rho)) {
        const double ir = rcp64(rho);
        ux = jx * ir;
        uy = jy * ir;
    } else {
        ux = jx / rho;
        uy = jy / rho;
    }
}

// FP64 storage: a cell's nine equilibria, from three factors along each axis,
// go to the slots that pull them (slot i of the cell at x - e_i, or the cell's
// own slot opp(i) where that is a wall or solid), so that each is evaluated
// once: about 40 FP64 operations a cell.  Evaluated per slot instead, from
// the neighbour's fields, 1024 x 1024 cells took 234 us (now 74 us).
template <bool MASK>
__global__ void __launch_bounds__(kThreads)
init_kernel(double* __restrict__ f, const AuxParams p, const double* __restrict__ rho,
            const double* __restrict__ ux, const double* __restrict__ uy) {
    const double iah2 = 0.5 / (p.a * p.a);
    LBM_FOR_ALL_CELLS(p, c) {
        const int y = row_of(p, c), x = (int)(c - (long long)y * p.nx);
        const long long o = (long long)y * p.rstride + x;
        const unsigned sb = link_bits<MASK>(p, x, y);
        if (sb == 0xFFu) {
#pragma unroll
            for (int i = 0; i < 9; ++i) f[i * p.plane + o] = 0.0;
            continue;
        }
        const double r = rho ? rho[c] : 1.0, u = ux ? ux[c] : 0.0, v = uy ? uy[c] : 0.0;
        double X[3], Y[3];  // e = 0, +1, -1
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            X[k] = r * phi_x<double>(k == 2 ? -1 : k, u, p.cs2);
            Y[k] = phi_y<double>(k == 2 ? -1 : k, v, p.cs2, p.a, iah2);
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const double v9 = X[ex(i) < 0 ? 2 : ex(i)] * Y[ey(i) < 0 ? 2 : ey(i)] - p.wrest[i];
            if (i > 0 && ((sb >> (i - 1)) & 1u)) {
                f[opp(i) * p.plane + o] = v9;
            } else {
                int tx = x - ex(i), ty = y - ey(i);
                tx = tx < 0 ? tx + p.nx : tx >= p.nx ? tx - p.nx : tx;
                ty = ty < 0 ? ty + p.ny : ty >= p.ny ? ty - p.ny : ty;
                f[i * p.plane + (long long)ty * p.rstride + tx] = v9;
            }
        }
    }
}

// FP32 storage: a block owns up to kThreads columns and marches down a band
// of rows, keeping the FP32 state (r - rho0, u, v) of the rows y - 1, y,
// y + 1 and of one column either side in shared memory, so that each cell's
// FP64 input is converted once rather than once per population.
//
// Bound by the latency of the FP64 reads, then by memory: the row after the
// next is fetched into registers while a row is written, and a ring of four
// rows needs one barrier a row (a row's slot is written again two barriers
// after its last read).  Small lattices take short bands (init_rows), so
// that a launch is not one block's march.
constexpr int kInitRows = 16;  // most rows of a band (more when ny / 16 > 65535)
constexpr int kInitThreads = kThreads + 32;  // one column a thread; a last warp for the two halo columns

template <bool MASK>
__global__ void __launch_bounds__(kInitThreads)
init32_kernel(float* __restrict__ f, const AuxParams p, const double* __restrict__ rho,
              const double* __restrict__ ux, const double* __restrict__ uy, int rows) {
    constexpr int SW = kThreads + 2;
    __shared__ float st[3][4][SW];  // [component][ring row][column x - x0 + 1]
    const Feq32 feq{p.cs232, p.a32, p.iah232, p.rho032};
    const int tx = threadIdx.x;
    const int x0 = blockIdx.x * kThreads;
    const int w = min(kThreads, p.nx - x0);
    const int y0 = blockIdx.y * rows;
    const int y1 = min(p.ny, y0 + rows);
    if (w <= 0 || y0 >= p.ny) return;
    // the ring column this thread fetches (-1: none): its own, or a halo one
    const int c = tx < w ? tx + 1 : tx == kThreads ? 0 : tx == kThreads + 1 ? w + 1 : -1;
    int gx = x0 - 1 + c;
    if (gx < 0) gx = p.px ? gx + p.nx : -1;
    else if (gx >= p.nx) gx = p.px ? gx - p.nx : -1;
    if (c < 0) gx = -1;
    double qr, qu, qv;
    auto fetch = [&](int yy) {  // outside a wall: the rest state, which nothing reads
        int gy = yy;
        if (gy < 0) gy = p.py ? gy + p.ny : -1;
        else if (gy >= p.ny) gy = p.py ? gy - p.ny : -1;
        qr = p.rho0;
        qu = qv = 0.0;
        if (gx < 0 || gy < 0) return;
        const long long t = (long long)gy * p.nx + gx;
        qr = rho ? rho[t] : 1.0;
        if (ux) qu = ux[t];
        if (uy) qv = uy[t];
    };
    auto slot = [&](int yy) { return (yy - y0 + 1) & 3; };
    auto put = [&](int yy) {
        if (c < 0) return;
        const int s = slot(yy);
        st[0][s][c] = narrow(qr - p.rho0);
        st[1][s][c] = narrow(qu);
        st[2][s][c] = narrow(qv);
    };
    fetch(y0 - 1);
    const double r0 = qr, u0 = qu, v0 = qv;
    fetch(y0);
    const double r1 = qr, u1 = qu, v1 = qv;
    fetch(y0 + 1);
    const double r2 = qr, u2 = qu, v2 = qv;
    qr = r0, qu = u0, qv = v0;
    put(y0 - 1);
    qr = r1, qu = u1, qv = v1;
    put(y0);
    qr = r2, qu = u2, qv = v2;
    for (int y = y0; y < y1; ++y) {
        put(y + 1);
        __syncthreads();
        if (y + 1 < y1) fetch(y + 2);
        if (tx >= w) continue;
        const int x = x0 + tx;
        const long long o = (long long)y * p.rstride + x;
        const unsigned sb = link_bits<MASK>(p, x, y);
        if (sb == 0xFFu) {
#pragma unroll
            for (int i = 0; i < 9; ++i) f[i * p.plane + o] = 0.0f;
            continue;
        }
        const int k = slot(y);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            float v;
            if (i > 0 && ((sb >> (opp(i) - 1)) & 1u)) {
                // pulled back by the cell itself
                v = feq(opp(i), st[0][k][c], st[1][k][c], st[2][k][c]);
            } else {
                const int kk = slot(y + ey(i)), cc = c + ex(i);
                v = feq(i, st[0][kk][cc], st[1][kk][cc], st[2][kk][cc]);
            }
            f[i * p.plane + o] = v;
        }
    }
}

// The same for narrow lattices, a cell a thread: each reads its nine neighbours' fields
// (from L1 and L2: a row is a few sectors) and evaluates the same expressions.  Up to
// 48 columns, where a block's march leaves most of its threads without a column, and
// from the rows on that make it march more than one (init_rows); us with obstacles,
// cells / march: 3 x 100000 23 / 199, 17 x 100000 78 / 238, 40 x 40000 64 / 113,
// 33 x 10000 19 / 28; but 33 x 1000 9.7 / 9.8, 17 x 1000 9.0 / 9.7 (without obstacles
// 9.6 / 8.6), 64 x 30000 without obstacles 68 / 59, 2049 x 2048 163 / 86.
constexpr int kInitNarrow = 48, kInitTall = 2432;
template <bool MASK>
__global__ void __launch_bounds__(kThreads)
init32_narrow_kernel(float* __restrict__ f, const AuxParams p, const double* __restrict__ rho,
                     const double* __restrict__ ux, const double* __restrict__ uy) {
    const Feq32 feq{p.cs232, p.a32, p.iah232, p.rho032};
    LBM_FOR_ALL_CELLS(p, c) {
        const int y = row_of(p, c), x = (int)(c - (long long)y * p.nx);
        const long long o = (long long)y * p.rstride + x;
        const unsigned sb = link_bits<MASK>(p, x, y);
        if (sb == 0xFFu) {
#pragma unroll
            for (int i = 0; i < 9; ++i) f[i * p.plane + o] = 0.0f;
            continue;
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            // the cell that pulls the slot, or this one as the opposite direction
            const bool back = i > 0 && ((sb >> (opp(i) - 1)) & 1u);
            const long long t = back || i == 0 ? c : target(p, x, y, i);
            const float dr = narrow((rho ? rho[t] : 1.0) - p.rho0);
            const float u = narrow(ux ? ux[t] : 0.0), v = narrow(uy ? uy[t] : 0.0);
            f[i * p.plane + o] = back ? feq(opp(i), dr, u, v) : feq(i, dr, u, v);
        }
    }
}

// Rows of an init32_kernel band: kInitRows where the blocks then fill the
// GPU (about eight 256-thread blocks on each of 152 SMs), fewer on smaller
// lattices, down to one.
int init_rows(int nx, int ny) {
    const long long segs = (nx + kThreads - 1) / kThreads;
    const long long fit = segs * ny / 1216;
    const int rows = (int)(fit < 1 ? 1 : fit < kInitRows ? fit : kInitRows);
    return max(rows, (ny + 65534) / 65535);  // grid.y limit
}

template <typename T>
__device__ __forceinline__ T stored(double v);
template <>
__device__ __forceinline__ float stored<float>(double v) { return narrow(v); }
template <>
__device__ __forceinline__ double stored<double>(double v) { return v; }

template <typename T, bool MASK>
__global__ void __launch_bounds__(kThreads)
set_f_kernel(T* __restrict__ f, const AuxParams p, const double* __restrict__ fin) {
    const long long N = (long long)p.nx * p.ny;
    LBM_FOR_ALL_CELLS(p, c) {
        const int y = row_of(p, c), x = (int)(c - (long long)y * p.nx);
        const long long o = (long long)y * p.rstride + x;
        const unsigned sb = link_bits<MASK>(p, x, y);
        if (sb == 0xFFu) {
#pragma unroll
            for (int i = 0; i < 9; ++i) f[i * p.plane + o] = T(0);
            continue;
        }
        double v[9];
#pragma unroll
        for (int i = 0; i < 9; ++i)
            v[i] = (i > 0 && ((sb >> (opp(i) - 1)) & 1u))
                       ? fin[opp(i) * N + c]
                       : fin[i * N + (i == 0 ? c : target(p, x, y, i))];
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i * p.plane + o] = stored<T>(v[i] - p.wrest[i]);
    }
}

// (six blocks an SM: at 44 registers, five, FP64 1000 x 1000 took 26.4 us, at 40 24.7)
template <typename T, bool MASK>
__global__ void __launch_bounds__(kThreads, 6)
get_f_kernel(const T* __restrict__ f, const AuxParams p, double* __restrict__ fout) {
    const long long N = (long long)p.nx * p.ny;
    LBM_FOR_ALL_CELLS(p, c) {
        const int y = row_of(p, c), x = (int)(c - (long long)y * p.nx);
        const unsigned sb = link_bits<MASK>(p, x, y);
        if (sb == 0xFFu) {
#pragma unroll
            for (int i = 0; i < 9; ++i) fout[i * N + c] = 0.0;
            continue;
        }
        T g[9];
        pull(f, p, x, y, sb, g);
#pragma unroll
        for (int i = 0; i < 9; ++i) fout[i * N + c] = widen(g[i]) + p.wrest[i];
    }
}

// rho, rho u (with half the force) and u of one fluid cell from its pulled
// deviations, in FP64.  fixed: the density deviation in fixed point, where
// the result is true.
struct Macro {
    double rho, jx, jy, ux, uy;
};
template <typename T>
__device__ __forceinline__ bool macro(const AuxParams& p, const T g[9], Macro& m,
                                      long long& fixed) {
    Raw r;
    const bool ok = raw_sums(g, r, fixed);
    m.rho = p.rho0 + r.d;
    m.jx = r.jx + 0.5 * p.Fx;
    m.jy = fma(p.a, r.jy, 0.5 * p.Fy);
    over_rho(m.rho, m.jx, m.jy, m.ux, m.uy);
    return ok;
}
__device__ __forceinline__ bool finite64(double v) {
    return ((unsigned)__double2hiint(v) & 0x7FF00000u) != 0x7FF00000u;
}

// The read-out of FP32 storage (lbm_moments): the nine deviations summed in
// FP32 and rho = rho0 + d formed in FP64, u in FP32 (the accuracy the FP32
// state holds), so that the FP64 pipe only converts.  The diagnostics and
// residuals keep the FP64 macro().
__device__ __forceinline__ void macro_out(const AuxParams& p, const float g[9], double& rho,
                                          double& ux, double& uy) {
    float d = 0.0f, jx = 0.0f, jy = 0.0f;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        d += g[i];
        if (ex(i) != 0) jx += ex(i) > 0 ? g[i] : -g[i];
        if (ey(i) != 0) jy += ey(i) > 0 ? g[i] : -g[i];
    }
    rho = p.rho0 + widen(d);
    const float r = p.rho032 + d;
    ux = widen((jx + p.hFx32) / r);
    uy = widen((p.a32 * jy + p.hFy32) / r);
}
__device__ __forceinline__ void macro_out(const AuxParams& p, const double g[9], double& rho,
                                          double& ux, double& uy) {
    Macro m;
    long long fixed;
    macro(p, g, m, fixed);
    rho = m.rho;
    ux = m.ux;
    uy = m.uy;
}

template <typename T, bool MASK>
__global__ void moments_kernel(const T* __restrict__ f, const AuxParams p,
                               double* rho, double* ux, double* uy) {
    LBM_FOR_CELLS(p) {
        const long long c = (long long)y * p.nx + x;
        const unsigned sb = link_bits<MASK>(p, x, y);
        double r = 0.0, u = 0.0, v = 0.0;
        if (sb != 0xFFu) {
            T g[9];
            pull(f, p, x, y, sb, g);
            macro_out(p, g, r, u, v);
        }
        if (rho) rho[c] = r;
        if (ux) ux[c] = u;
        if (uy) uy[c] = v;
    }
}

// The density of every cell in FP64 (0 in a solid cell), for the stress.
template <typename T, bool MASK>
__global__ void __launch_bounds__(kThreads)
density_kernel(const T* __restrict__ f, const AuxParams p, double* __restrict__ rho) {
    LBM_FOR_ALL_CELLS(p, c) {
        const int y = row_of(p, c), x = (int)(c - (long long)y * p.nx);
        const unsigned sb = link_bits<MASK>(p, x, y);
        double r = 0.0;
        if (sb != 0xFFu) {
            T g[9];
            pull(f, p, x, y, sb, g);
            Raw s;
            long long fixed;
            raw_sums(g, s, fixed);
            r = p.rho0 + s.d;
        }
        rho[c] = r;
    }
}

// Local strain rates of one fluid cell from its raw non-equilibrium moments
// (Eq. 34-40; the left side of Eq. 39 read as d_y u_x + d_x u_y) and the
// viscous stress of the recovered Navier-Stokes equations (Eq. 30-33), all in
// FP64.  The density gradient is the central difference of the step (spacing
// 2 along x and 2a along y), a wall or solid neighbour counting with the
// cell's own density.
// Bound by the FP64 lanes: about 60 operations a cell, with the moments as
// deviations from the rest state (the rest part cancels analytically), two
// reciprocals and products in place of the five divisions, and the constants
// from the host.
struct StressConst {
    double a, a2, cs2, g1, g2, hFx, hFy;
    double bc, cb, d, v, dv;  // (b1 + c1)/2, (c2 - b2)/2, (b1 - c1)/2, (b2 + c2)/2, d v
    double e5, k5;            // xy strain rate and stress over the xy moment
    double sp, sm;            // bulk plus and minus shear viscosity
};
template <typename T, bool MASK>
__global__ void __launch_bounds__(kThreads)
stress_kernel(const T* __restrict__ f, const AuxParams p, const StressConst q,
              const double* __restrict__ rho,
              double* __restrict__ dxux, double* __restrict__ dyuy, double* __restrict__ sxy,
              double* __restrict__ txx, double* __restrict__ tyy, double* __restrict__ txy) {
    LBM_FOR_ALL_CELLS(p, c) {
        const int y = row_of(p, c), x = (int)(c - (long long)y * p.nx);
        const long long row = c - x;
        const unsigned sb = link_bits<MASK>(p, x, y);
        double e_xx = 0.0, e_yy = 0.0, e_xy = 0.0, s_xx = 0.0, s_yy = 0.0, s_xy = 0.0;
        if (sb != 0xFFu) {
            T g[9];
            pull(f, p, x, y, sb, g);
            const int xm = x == 0 ? p.nx - 1 : x - 1, xp = x == p.nx - 1 ? 0 : x + 1;
            const int ym = y == 0 ? p.ny - 1 : y - 1, yp = y == p.ny - 1 ? 0 : y + 1;
            const double rc = rho[c];
            const double rW = (sb & 1u) ? rc : rho[row + xm];
            const double rS = (sb & 2u) ? rc : rho[(long long)ym * p.nx + x];
            const double rE = (sb & 4u) ? rc : rho[row + xp];
            const double rN = (sb & 8u) ? rc : rho[(long long)yp * p.nx + x];
            Raw s;
            long long fixed;
            raw_sums(g, s, fixed);
            const double r = p.rho0 + s.d;
            const double ir = rcp64_ok(r) ? rcp64(r) : 1.0 / r;
            const double jx = s.jx + q.hFx, jy = fma(q.a, s.jy, q.hFy);
            const double ux = jx * ir, uy = jy * ir;
            // non-equilibrium second-order moments m - m^eq, and the gradient terms
            const double n20 = fma(-jx, ux, fma(-q.cs2, s.d, s.sxx));
            const double n02 = fma(-jy, uy, fma(-q.cs2, s.d, q.a2 * s.syy));
            const double n11 = fma(-jx, uy, q.a * s.sxy);
            const double m20 = fma(q.g1 * ux, rE - rW, n20), m02 = fma(q.g2 * uy, rN - rS, n02);
            // With B1 = 3/2 ux^2 + b1, C1 = 3/2 ux^2 + c1, B2 = 3/2 uy^2 + b2, C2 = c2 -
            // 3/2 uy^2, the strain rates are
            //   rho dx ux = (C2 R3 - B2 R4) / det, rho dy uy = (B1 R4 - C1 R3) / det,
            //   R3 = m20 + m02, R4 = m20 - m02, det = B1 C2 - B2 C1;
            // in halves of sums and differences of the coefficients the products
            // that cancel are gone (8 of 22 FP64 operations).
            const double P = fma(1.5, ux * ux, q.bc), Q = fma(-1.5, uy * uy, q.cb);
            const double det = fma(P, Q, q.dv);
            const double id = rcp64_ok(det) ? rcp64(det) : 1.0 / det;
            const double rxx = fma(Q, m20, q.v * m02) * id, ryy = fma(q.d, m20, -(P * m02)) * id;
            e_xx = rxx * ir;
            e_yy = ryy * ir;
            e_xy = q.e5 * n11 * ir;
            s_xx = fma(q.sp, rxx, q.sm * ryy);
            s_yy = fma(q.sm, rxx, q.sp * ryy);
            s_xy = q.k5 * n11;
        }
        if (dxux) dxux[c] = e_xx;
        if (dyuy) dyuy[c] = e_yy;
        if (sxy) sxy[c] = e_xy;
        if (txx) txx[c] = s_xx;
        if (tyy) tyy[c] = s_yy;
        if (txy) txy[c] = s_xy;
    }
}

// Adds v exactly (down to 2^-kMassShift) to a fixed-point number held as
// 24-bit limbs.  Returns false when v is too large for the accumulator (32 or more
// in magnitude) or not finite.
__device__ __forceinline__ bool add_fixed(long long limb[kMassLimbs], double v) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
    const int E = (int)((bits >> 52) & 0x7FF);
    unsigned long long M = bits & 0xFFFFFFFFFFFFFull;
    if (E == 0x7FF) return false;
    int e2;
    if (E == 0) e2 = -1074;
    else { M |= 1ull << 52; e2 = E - 1075; }
    if (M == 0) return true;
    int pos = e2 + kMassShift;
    if (pos < 0) {
        if (pos <= -64) return true;   // below the accumulator's resolution
        M >>= -pos;
        pos = 0;
    }
    if (pos > 24 * (kMassLimbs - 4)) return false;
    const int k0 = pos / 24, o = pos % 24;
    const unsigned __int128 t = (unsigned __int128)M << o;
    long long c[4] = {(long long)(t & 0xFFFFFF), (long long)((t >> 24) & 0xFFFFFF),
                      (long long)((t >> 48) & 0xFFFFFF), (long long)(t >> 72)};
    const bool neg = (bits >> 63) != 0;
#pragma unroll
    for (int k = 0; k < kMassLimbs; ++k) {
        const int j = k - k0;
        long long add = 0;
        if (j == 0) add = c[0];
        else if (j == 1) add = c[1];
        else if (j == 2) add = c[2];
        else if (j == 3) add = c[3];
        limb[k] += neg ? -add : add;
    }
    return true;
}

// The mass of a thread's cells as one 128-bit integer, where every value is
// an exact multiple of the integer's unit; the rest goes through add_fixed.
// FP32 storage: the sum of a cell's deviations in units of 2^-kFixedShift.
__device__ __forceinline__ bool add_mass(__int128& acc, long long limb[kMassLimbs],
                                         const float g[9], bool exact, long long fixed) {
    if (exact) {
        acc += fixed;
        return true;
    }
    bool ok = true;
#pragma unroll
    for (int i = 0; i < 9; ++i) ok &= add_fixed(limb, (double)g[i]);
    return ok;
}
// FP64 storage: each deviation in units of 2^-100, where it is between 2^-48 and
// 2^5 in magnitude, which is also where add_fixed ends (a cell with a larger one
// stays out of every sum); below 2^19 values a thread: < 2^124.
__device__ __forceinline__ bool add_mass(__int128& acc, long long limb[kMassLimbs],
                                         const double g[9], bool, long long) {
    bool ok = true;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(g[i]);
        const int sh = (int)((b >> 52) & 0x7FF) - 975;  // exponent - 1075 + 100
        if (sh >= 0 && sh < 1028 - 975) {
            const __int128 v = (__int128)((b & 0xFFFFFFFFFFFFFull) | (1ull << 52)) << sh;
            acc += (long long)b < 0 ? -v : v;
        } else {
            ok &= add_fixed(limb, g[i]);
        }
    }
    return ok;
}
// Spreads a 128-bit integer in units of 2^-58 (FP32) or 2^-100 (FP64) over
// the 24-bit limbs.
template <typename T>
__device__ __forceinline__ void spread(__int128 acc, long long limb[kMassLimbs]) {
    constexpr int kBit = kMassShift - (sizeof(T) == 4 ? kFixedShift : 100);
    constexpr int k0 = kBit / 24, o = kBit % 24;
    limb[k0] += (long long)(acc & ((1 << (24 - o)) - 1)) << o;
    acc >>= 24 - o;
#pragma unroll
    for (int k = k0 + 1; k < kMassLimbs - 1; ++k) {
        limb[k] += (long long)(acc & 0xFFFFFF);
        acc >>= 24;
    }
    limb[kMassLimbs - 1] += (long long)acc;
}

template <typename V>
__device__ __forceinline__ V warp_sum(V v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    return v;
}

// Sums one DiagPartial per thread over the block in a fixed order: over each
// warp by shuffles, then one thread per field over the warps.
__device__ void block_reduce(DiagPartial& d, DiagPartial* out) {
    constexpr int kWarps = kThreads / 32;
    __shared__ DiagPartial sh[kWarps];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    d.mx = warp_sum(d.mx);
    d.my = warp_sum(d.my);
    d.en = warp_sum(d.en);
    d.dres = warp_sum(d.dres);
    d.ures = warp_sum(d.ures);
    d.sres = warp_sum(d.sres);
    d.nonfinite = warp_sum(d.nonfinite);
#pragma unroll
    for (int k = 0; k < kMassLimbs; ++k) d.limb[k] = warp_sum(d.limb[k]);
    if (lane == 0) sh[w] = d;
    __syncthreads();
    const int k = threadIdx.x;
    double* real = &out->mx;
    long long* whole = &out->nonfinite;
    if (k < kDiagReals) {
        double s = (&sh[0].mx)[k];
        for (int i = 1; i < kWarps; ++i) s += (&sh[i].mx)[k];
        real[k] = s;
    } else if (k < kDiagReals + 1 + kMassLimbs) {
        long long s = 0;
        for (int i = 0; i < kWarps; ++i) s += (&sh[i].nonfinite)[k - kDiagReals];
        whole[k - kDiagReals] = s;
    }
}

// The steady residual is taken on the two-step mean velocity
// ubar(n) = (u(n) + u(n-1)) / 2 when the state one step earlier is at hand
// (fprev, the other buffer): the scheme carries exact invariants, the
// staggered momenta sum (-1)^(x+n) rho ux and sum (-1)^(y+n) rho uy, whose
// motion alternates sign every step; a residual between two states an even
// number of steps apart never sees it, and the mean cancels it.  The
// step-to-step change |u(n) - u(n-1)|^2 is summed beside it.
template <typename T, bool MASK>
__global__ void __launch_bounds__(kThreads)
diag_kernel(const T* __restrict__ f, const T* __restrict__ fprev, const AuxParams p,
            double* __restrict__ uprev, int have_prev, DiagPartial* part) {
    const long long N = (long long)p.nx * p.ny;
    DiagPartial d = {};
    __int128 acc = 0;
    LBM_FOR_ALL_CELLS(p, c) {
        const int y = row_of(p, c), x = (int)(c - (long long)y * p.nx);
        const unsigned sb = link_bits<MASK>(p, x, y);
        if (sb == 0xFFu) continue;
        // every read first: one latency a cell
        T g[9], q[9];
        double pu = 0.0, pv = 0.0;
        pull(f, p, x, y, sb, g);
        if (fprev) pull(fprev, p, x, y, sb, q);
        if (have_prev) {
            pu = uprev[c];
            pv = uprev[N + c];
        }
        Macro m;
        long long fixed;
        const bool exact = macro(p, g, m, fixed);
        const bool ok = add_mass(acc, d.limb, g, exact, fixed);
        if (!ok || !finite64(m.rho) || !finite64(m.ux) || !finite64(m.uy)) {
            d.nonfinite += 1;
            continue;
        }
        d.mx += m.jx;
        d.my += m.jy;
        d.en = fma(0.5, fma(m.jx, m.ux, m.jy * m.uy), d.en);
        double mx = m.ux, my = m.uy;
        if (fprev) {
            Macro m1;
            macro(p, q, m1, fixed);
            const double sx = m.ux - m1.ux, sy = m.uy - m1.uy;
            d.sres = fma(sx, sx, fma(sy, sy, d.sres));
            mx = 0.5 * (m.ux + m1.ux);
            my = 0.5 * (m.uy + m1.uy);
        }
        d.ures = fma(mx, mx, fma(my, my, d.ures));
        if (have_prev) {
            const double du = mx - pu, dv = my - pv;
            d.dres = fma(du, du, fma(dv, dv, d.dres));
        }
        uprev[c] = mx;
        uprev[N + c] = my;
    }
    spread<T>(acc, d.limb);
    block_reduce(d, part + blockIdx.x);
}

// Sums the n partials into *out, beside the step kernels' status word (so
// that the host reads one result).
__global__ void __launch_bounds__(kThreads)
diag_final(const DiagPartial* part, int n, const int* status, DiagPartial* out) {
    DiagPartial d = {};
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const DiagPartial& q = part[i];
        d.mx += q.mx;
        d.my += q.my;
        d.en += q.en;
        d.dres += q.dres;
        d.ures += q.ures;
        d.sres += q.sres;
        d.nonfinite += q.nonfinite;
#pragma unroll
        for (int k = 0; k < kMassLimbs; ++k) d.limb[k] += q.limb[k];
    }
    block_reduce(d, out);
    if (threadIdx.x == 0) out->status = *status;
}

// Residual sums of one thread summed over the block, in a fixed order.
__device__ void res_block_reduce(ResPartial& d, ResPartial* out) {
    __shared__ ResPartial sh[kThreads / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    d.dres = warp_sum(d.dres);
    d.ures = warp_sum(d.ures);
    d.nonfinite = warp_sum(d.nonfinite);
    if (lane == 0) sh[w] = d;
    __syncthreads();
    if (threadIdx.x == 0) {
        ResPartial s = sh[0];
        for (int i = 1; i < (int)(blockDim.x / 32); ++i) {
            s.dres += sh[i].dres;
            s.ures += sh[i].ures;
            s.nonfinite += sh[i].nonfinite;
        }
        *out = s;
    }
}

// Block w sums reduction chunk w - rbegin[j] of active lattice j: its runs of
// kThreads cells chunk, chunk + nchunk, ...
__global__ void __launch_bounds__(kThreads)
batch_res_kernel(const BatchLattice<float>* __restrict__ lat, const BatchAux* __restrict__ aux,
                 const int* __restrict__ active, const int* __restrict__ rbegin,
                 const int* __restrict__ counts, const int* __restrict__ two, int parity,
                 ResPartial* part) {
    const int n = counts[0];
    const int w = blockIdx.x;
    if (w >= counts[1]) return;
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (rbegin[mid] <= w) lo = mid;
        else hi = mid - 1;
    }
    const int k = active[lo];
    const BatchAux& B = aux[k];
    const AuxParams& p = B.a;
    const float* f = lat[k].f[parity];
    const float* fp = two[k] ? lat[k].f[parity ^ 1] : nullptr;  // one step earlier
    const int chunk = w - rbegin[lo];
    const long long N = (long long)p.nx * p.ny;
    double* __restrict__ up = B.uprev;
    ResPartial d = {};
    for (long long c = chunk * (long long)kThreads + threadIdx.x; c < N;
         c += B.nchunk * (long long)kThreads) {
        const int y = row_of(p, c), x = (int)(c - (long long)y * p.nx);
        const unsigned sb = link_bits<true>(p, x, y);
        if (sb == 0xFFu) continue;
        float g[9], q[9];
        pull(f, p, x, y, sb, g);
        if (fp) pull(fp, p, x, y, sb, q);
        const double pu = up[c], pv = up[N + c];
        Macro m;
        long long fixed;
        macro(p, g, m, fixed);
        if (!finite64(m.rho) || !finite64(m.ux) || !finite64(m.uy)) {
            d.nonfinite += 1;
            continue;
        }
        double mx = m.ux, my = m.uy;  // the two-step mean velocity, as in diag_kernel
        if (fp) {
            Macro m1;
            macro(p, q, m1, fixed);
            mx = 0.5 * (m.ux + m1.ux);
            my = 0.5 * (m.uy + m1.uy);
        }
        const double du = mx - pu, dv = my - pv;
        d.dres = fma(du, du, fma(dv, dv, d.dres));
        d.ures = fma(mx, mx, fma(my, my, d.ures));
        up[c] = mx;
        up[N + c] = my;
    }
    res_block_reduce(d, part + B.pbegin + chunk);
}

// Block j sums the chunks of active lattice j in chunk order.
__global__ void __launch_bounds__(kThreads)
batch_res_final(const BatchAux* __restrict__ aux, const int* __restrict__ active,
                const int* __restrict__ counts, const ResPartial* __restrict__ part,
                ResPartial* out) {
    if ((int)blockIdx.x >= counts[0]) return;
    const int k = active[blockIdx.x];
    const BatchAux& B = aux[k];
    ResPartial d = {};
    for (int i = threadIdx.x; i < B.nchunk; i += blockDim.x) {
        const ResPartial& q = part[B.pbegin + i];
        d.dres += q.dres;
        d.ures += q.ures;
        d.nonfinite += q.nonfinite;
    }
    res_block_reduce(d, out + k);
}

// blocks of LBM_FOR_ALL_CELLS, at most `most`
int cell_grid(const AuxParams& p, int most = 4096) {
    const long long n = ((long long)p.nx * p.ny + kThreads - 1) / kThreads;
    return n < most ? (int)n : most;
}

// grid of LBM_FOR_CELLS: blocks across a row, rows down the grid, at most
// 16384 blocks
dim3 grid2_for(int nx, int ny) {
    const int gx = (nx + kThreads - 1) / kThreads;
    const int gy = ny < 16384 / gx ? ny : (16384 / gx > 0 ? 16384 / gx : 1);
    return dim3(gx > 0 ? gx : 1, gy > 0 ? gy : 1);
}

}  // namespace

template <typename T>
cudaError_t launch_init(T* f, const AuxParams& p, const double* rho, const double* ux,
                        const double* uy, cudaStream_t s) {
    if constexpr (sizeof(T) == 4) {
        if (p.nx <= kInitNarrow && p.ny >= kInitTall) {
            const int g = cell_grid(p);
            if (p.lmask) init32_narrow_kernel<true><<<g, kThreads, 0, s>>>(f, p, rho, ux, uy);
            else init32_narrow_kernel<false><<<g, kThreads, 0, s>>>(f, p, rho, ux, uy);
            return cudaGetLastError();
        }
        const int rows = init_rows(p.nx, p.ny);
        const dim3 g((p.nx + kThreads - 1) / kThreads, (p.ny + rows - 1) / rows);
        if (p.lmask) init32_kernel<true><<<g, kInitThreads, 0, s>>>(f, p, rho, ux, uy, rows);
        else init32_kernel<false><<<g, kInitThreads, 0, s>>>(f, p, rho, ux, uy, rows);
    } else {
        const int g = cell_grid(p);
        if (p.lmask) init_kernel<true><<<g, kThreads, 0, s>>>(f, p, rho, ux, uy);
        else init_kernel<false><<<g, kThreads, 0, s>>>(f, p, rho, ux, uy);
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_set_f(T* f, const AuxParams& p, const double* fin, cudaStream_t s) {
    const int g = cell_grid(p);
    if (p.lmask) set_f_kernel<T, true><<<g, kThreads, 0, s>>>(f, p, fin);
    else set_f_kernel<T, false><<<g, kThreads, 0, s>>>(f, p, fin);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_get_f(const T* f, const AuxParams& p, double* fout, cudaStream_t s) {
    const int g = cell_grid(p);
    if (p.lmask) get_f_kernel<T, true><<<g, kThreads, 0, s>>>(f, p, fout);
    else get_f_kernel<T, false><<<g, kThreads, 0, s>>>(f, p, fout);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_moments(const T* f, const AuxParams& p, double* rho, double* ux,
                           double* uy, cudaStream_t s) {
    const dim3 g = grid2_for(p.nx, p.ny);
    if (p.lmask) moments_kernel<T, true><<<g, kThreads, 0, s>>>(f, p, rho, ux, uy);
    else moments_kernel<T, false><<<g, kThreads, 0, s>>>(f, p, rho, ux, uy);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_density(const T* f, const AuxParams& p, double* rho, cudaStream_t s) {
    const int g = cell_grid(p);
    if (p.lmask) density_kernel<T, true><<<g, kThreads, 0, s>>>(f, p, rho);
    else density_kernel<T, false><<<g, kThreads, 0, s>>>(f, p, rho);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_stress(const T* f, const AuxParams& p, const double* rho, double* dxux,
                          double* dyuy, double* sxy, double* txx, double* tyy, double* txy,
                          cudaStream_t s) {
    const int g = cell_grid(p);
    const double a2 = p.a * p.a, c = p.cs2;
    StressConst q;
    q.a = p.a;
    q.a2 = a2;
    q.cs2 = c;
    const double nu4 = c * (1.0 / p.w4 - 0.5), nu5 = c * (1.0 / p.w5 - 0.5),
                 zeta = c * (1.0 / p.w3 - 0.5);
    const double b1 = -2.0 * c / p.w3 - 0.5 * (1.0 - 3.0 * c);
    const double b2 = -2.0 * c / p.w3 - 0.5 * (a2 - 3.0 * c);
    const double c1 = -2.0 * c / p.w4 - 0.5 * (1.0 - 3.0 * c);
    const double c2 = 2.0 * c / p.w4 + 0.5 * (a2 - 3.0 * c);
    q.bc = 0.5 * (b1 + c1);
    q.cb = 0.5 * (c2 - b2);
    q.d = 0.5 * (b1 - c1);
    q.v = 0.5 * (b2 + c2);
    q.dv = q.d * q.v;
    q.g1 = 0.25 * (1.0 - 3.0 * c);           // with the spacing 2 of the differences
    q.g2 = 0.25 * (a2 - 3.0 * c) / p.a;      // and 2a
    q.e5 = -p.w5 / c;
    q.k5 = nu5 * q.e5;
    q.sp = zeta + nu4;
    q.sm = zeta - nu4;
    q.hFx = 0.5 * p.Fx;
    q.hFy = 0.5 * p.Fy;
    if (p.lmask)
        stress_kernel<T, true><<<g, kThreads, 0, s>>>(f, p, q, rho, dxux, dyuy, sxy, txx, tyy, txy);
    else
        stress_kernel<T, false><<<g, kThreads, 0, s>>>(f, p, q, rho, dxux, dyuy, sxy, txx, tyy, txy);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_diag(const T* f, const T* fprev, const AuxParams& p, double* uprev,
                        int have_prev, DiagPartial* part, int nblocks, const int* status,
                        cudaStream_t s) {
    const int n = cell_grid(p, nblocks);
    if (p.lmask)
        diag_kernel<T, true><<<n, kThreads, 0, s>>>(f, fprev, p, uprev, have_prev, part);
    else
        diag_kernel<T, false><<<n, kThreads, 0, s>>>(f, fprev, p, uprev, have_prev, part);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    diag_final<<<1, kThreads, 0, s>>>(part, n, status, part + nblocks);
    return cudaGetLastError();
}

cudaError_t launch_batch_residual(const BatchLattice<float>* lat, const BatchAux* aux,
                                  const int* active, const int* rbegin, const int* counts,
                                  const int* two, int parity, ResPartial* part,
                                  ResPartial* out, int nactive, int nblocks, cudaStream_t s) {
    if (nactive <= 0 || nblocks <= 0) return cudaSuccess;
    batch_res_kernel<<<nblocks, kThreads, 0, s>>>(lat, aux, active, rbegin, counts, two, parity,
                                                  part);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    batch_res_final<<<nactive, kThreads, 0, s>>>(aux, active, counts, part, out);
    return cudaGetLastError();
}

#define LBM_AUX_INST(T)                                                                \
    template cudaError_t launch_init<T>(T*, const AuxParams&, const double*,          \
                                        const double*, const double*, cudaStream_t);  \
    template cudaError_t launch_set_f<T>(T*, const AuxParams&, const double*,         \
                                         cudaStream_t);                               \
    template cudaError_t launch_get_f<T>(const T*, const AuxParams&, double*,         \
                                         cudaStream_t);                               \
    template cudaError_t launch_moments<T>(const T*, const AuxParams&, double*,       \
                                           double*, double*, cudaStream_t);           \
    template cudaError_t launch_density<T>(const T*, const AuxParams&, double*,       \
                                           cudaStream_t);                             \
    template cudaError_t launch_stress<T>(const T*, const AuxParams&, const double*,  \
                                          double*, double*, double*, double*, double*, \
                                          double*, cudaStream_t);                     \
    template cudaError_t launch_diag<T>(const T*, const T*, const AuxParams&, double*, int, \
                                        DiagPartial*, int, const int*, cudaStream_t);
LBM_AUX_INST(float)
LBM_AUX_INST(double)

}  // namespace lbm
