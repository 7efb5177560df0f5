// Binary64 substep with exact integer stencil sums and fixed-point products
// (periodic grids).
//
// GB300 executes two FP64 lanes per SM per cycle: an FP64-pipe instruction holds
// its sub-partition's pipe for about 78 cycles per warp, a 64-bit integer addition
// for 2.3 and a 32 x 32 + 64 multiply-add for 2.2 (measured), so the binary64
// substep is bound by its FP64 instruction count.  Each field is first written
// as int64 fixed point about an offset of its own, F = round((f - c) 2^(b - E)),
// with c the midpoint of the field's range and 2^E above its half-range.  Every
// weight set of Eq. 13 sums to zero, so the offset changes no derivative.
//
// A plan picks one of three forms per substep from the fields' ranges,
// on the device (no host round trip):
//  * FX_GROUP (b = 56): the exponents E of the three components of u (and of A)
//    lie within FX_GROUP_SLACK binades of each other and share the largest as one
//    scale (a component keeps at least 50 bits of its own range).  Stencil
//    numerators are exact integers, the products of the right-hand side (u . grad,
//    S . grad ln rho, S : S, j x B, j^2, u x B) exact integer dot products
//    (fx_arith.cuh), the exponentials fixed point; what remains on the FP64 pipe
//    is a multiply-add or two per term of Eqs. B.1-B.4 and the Runge-Kutta update (62
//    instructions per cell).  Thin boxes (fx_form) go column by column over copies
//    without a halo instead, with b = 50, one binade of slack and binary64 products.
//  * FX_FIELD (b = 50): some component lies further below its group's largest, so
//    every field keeps its own scale; integer numerators are converted one by one
//    and the sums across components (curl A, grad(div u), grad(div A)) and the
//    products run in binary64 -- a component far smaller than the others (a
//    near-2-D flow, a weak field component) is resolved to 2^-50 of its own range.
//    States beyond the ranges FX_GROUP is sized for take it too: exponents
//    outside +-200, a mean flow 2^4 times its range, a uniform component of u far below
//    the others, |ln rho| or |xi| over 64 (with unequal spacing FX_PLAIN takes them).
//  * FX_PLAIN: a NaN or infinity in the state, or a range outside
//    [2^-960, 2^960): the substep runs plain binary64 stencils, exactly what
//    AC_STENCIL_FP64 computes (so a non-finite value propagates as in the
//    definition and shows in the step's CFL word).
#pragma once

#include <cuda.h>

#include <type_traits>

#include "fx_arith.cuh"
#include "substep.cuh"

namespace ac {

constexpr int FX_BITS = 56;        // b of FX_GROUP: 110 |F| (first derivatives) stays in 63 bits
constexpr int FX_FIELD_BITS = 50;  // b of FX_FIELD: 6744 |F| (sums of numerators) does
constexpr int FX_GROUP_SLACK = 6;  // binades a component may lie below its group's largest
constexpr int FX_MODE_SLACK = 1;   // the same, for the mode that ac_get_stencil_modes counts
constexpr int FX_EMAX = 200;       // |E| of FX_GROUP: products of two scales stay normal
enum { FX_GROUP = 0, FX_FIELD = 1, FX_PLAIN = 2 };

// Field -> group: 0 = ln rho, 1 = u, 2 = s, 3 = A.
__host__ __device__ __forceinline__ int fx_group(int q) {
    return q == 0 ? 0 : (q < 4 ? 1 : (q == 4 ? 2 : 3));
}

// Order-preserving map of binary64 bits to unsigned keys (NaNs sort beyond the
// infinities of their sign) and back.
__device__ __forceinline__ unsigned long long fx_key(unsigned long long b) {
    // negatives: every bit flipped; positives: the sign bit set
    return b ^ ((unsigned long long)((long long)b >> 63) | 0x8000000000000000ull);
}
__device__ __forceinline__ double fx_unkey(unsigned long long k) {
    return __longlong_as_double((long long)((k >> 63) ? (k & 0x7fffffffffffffffull) : ~k));
}

// round(v 2^s) modulo 2^64 for the binary64 v held in `b` (round half away from
// zero), by integer operations on the bits.  Two such values within 2^63 of each
// other subtract exactly in wrapping 64-bit arithmetic, however large each is.
__device__ __forceinline__ unsigned long long fx_round_grid(unsigned long long b, int s) {
    const int eb = (int)((b >> 52) & 0x7ff);
    unsigned long long m = b & 0xfffffffffffffull;
    int ex = -1074;
    if (eb != 0) {
        m |= 1ull << 52;
        ex = eb - 1075;
    }
    const int sh = ex + s;  // |v| 2^s = m 2^sh
    unsigned long long a;
    if (sh >= 0) {
        a = sh < 64 ? m << sh : 0ull;
    } else {
        const int k = -sh;
        a = k < 64 ? (m + (1ull << (k - 1))) >> k : 0ull;
    }
    return (b >> 63) ? 0ull - a : a;
}

// The int64 copies: eight arrays back to back, each padded by the radius-3 periodic
// halo (which the quantisation writes), so that the tensor memory accelerator can
// fetch any tile with its halo as one box; without the halo (halo = 0) for the boxes
// that go column by column.
struct FxPtrs {
    const double *f[NF];
    long long *F[NF];
    int halo;
    int py;  // rows of a plane
    Geom g;  // of the copies: with the halo px = nx + 6 made even (16-byte strides)
};

// The quantisation plan of one substep (device memory, written by
// fx_stats_kernel, read by the quantisation and substep kernels).
struct FxPlan {
    int kern;                  // the kernel that runs: FX_GROUP, FX_FIELD or FX_PLAIN
    int zero[NF];              // constant field: F = 0
    int s[NF];                 // F = round((f - c) 2^s), s = b - E
    unsigned long long C[NF];  // round(c 2^s) modulo 2^64
    unsigned long long taken[3];  // substeps counted in each mode (cumulative)
    unsigned long long ran[4];    // substeps that each form ran (AC_STENCIL_FORM_*, cumulative)
};

// One warp: lane q < NF plans field q (offset, exponent), then the lanes agree
// on the kernel.  Thread 0 also counts the substep under its mode: plain,
// per-field (a component more than one binade below its group's largest) or group.
__device__ __forceinline__ void fx_plan(unsigned long long *stats, FxPlan *plan, double gamma_cp,
                                        double gm1, int form) {
    const int q = threadIdx.x;
    int bad = 0, zero = 1, e = -100000, ec = -100000;
    double c = 0.0, big = 0.0;
    if (q < NF) {
        const double hi = fx_unkey(__ldcg(&stats[q])), lo = fx_unkey(__ldcg(&stats[NF + q]));
        stats[q] = 0ull;        // ready for the next substep's extremes
        stats[NF + q] = ~0ull;
        if (!isfinite(hi) || !isfinite(lo)) {
            bad = 1;
        } else {
            c = 0.5 * lo + 0.5 * hi;
            big = fmax(fabs(hi), fabs(lo));
            const double r = fmax(hi - c, c - lo);
            if (r > 0.0) {
                zero = 0;
                if (!(r >= 0x1p-960 && r < 0x1p960))
                    bad = 1;
                else  // smallest E with r < 2^E
                    e = (int)((__double_as_longlong(r) >> 52) & 0x7ff) - 1022;
            }
            if (c != 0.0)  // |c| < 2^ec
                ec = (int)((__double_as_longlong(c) >> 52) & 0x7ff) - 1022;
        }
    }
    // largest exponent of the field's group over its non-constant members (over
    // the offsets where every member is constant)
    const int g = q < NF ? fx_group(q) : -1;
    int eg = -100000, egc = -100000;
#pragma unroll
    for (int r = 0; r < NF; ++r) {
        const int er = __shfl_sync(0xffffffffu, e, r), cr = __shfl_sync(0xffffffffu, ec, r);
        if (fx_group(r) == g) {
            eg = er > eg ? er : eg;
            egc = cr > egc ? cr : egc;
        }
    }
    if (eg == -100000) eg = egc > -100000 ? egc : 0;
    const int any_bad = __any_sync(0xffffffffu, bad);
    const int far = __any_sync(0xffffffffu, q < NF && !zero && e < eg - FX_MODE_SLACK);
    // what FX_GROUP is sized for: the slack, the exponents, |u| < 2^(E + 4) (u is taken
    // from F + C, so that a constant component has to lie within the slack too, or be
    // zero), |ln rho| and |xi| below 64 (the fixed-point exp)
    const double xb = gamma_cp * __shfl_sync(0xffffffffu, big, 4) +
                      fabs(gm1) * __shfl_sync(0xffffffffu, big, 0);
    int out = q < NF && ((!zero && e < eg - FX_GROUP_SLACK) || eg > FX_EMAX || eg < -FX_EMAX);
    if (g == 1) out |= ec > eg + 4 || (zero && c != 0.0 && ec < eg - FX_GROUP_SLACK);
    if (q == 0) out |= !(big < 64.0) || !(xb < 64.0);
    const int any_out = __any_sync(0xffffffffu, out);
    // (FX_FIELD wants equal spacing: without it the plain stencils take its place; the
    // columns' FX_GROUP has binary64 products and only asks for the narrower slack)
    const int mode = any_bad ? FX_PLAIN : (far ? FX_FIELD : FX_GROUP);
    const int kern = form == FX_COLUMNS ? mode
                     : any_bad || (form == FX_UNEQUAL && any_out) ? FX_PLAIN
                     : any_out ? FX_FIELD : FX_GROUP;
    int s = FX_FIELD_BITS - (e > -100000 ? e : 0);
    if (kern == FX_GROUP) s = form == FX_COLUMNS ? FX_FIELD_BITS - eg : FX_BITS - eg;
    if (q < NF) {
        plan->zero[q] = zero;
        plan->s[q] = s;
        plan->C[q] = fx_round_grid((unsigned long long)__double_as_longlong(c), s);
    }
    if (q == 0) {
        plan->kern = kern;
        plan->ran[kern == FX_PLAIN   ? AC_STENCIL_FORM_PLAIN
                  : kern == FX_FIELD ? AC_STENCIL_FORM_FIELD
                  : form == FX_COLUMNS ? AC_STENCIL_FORM_GROUP : AC_STENCIL_FORM_PRODUCTS] += 1ull;
        if (form != FX_UNEQUAL) plan->taken[mode] += 1ull;
    }
}

// Per-field extremes of the current state: stats[q] = largest key of field q,
// stats[NF + q] = its smallest key.  Two cells per thread and iteration (16-byte
// loads; the arrays are 16-byte aligned), one CTA-wide reduction, then 16 atomics per
// CTA.  The last CTA to finish (stats[2 NF] counts them) makes the plan of them and
// resets the words for the next substep: as a kernel of its own the plan was 5 us of a
// 32^3 substep's 42.
__global__ void __launch_bounds__(256) fx_stats_kernel(FxPtrs p, long long n, unsigned long long *stats,
                                                       FxPlan *plan, double gamma_cp, double gm1,
                                                       int form) {
    unsigned long long hi[NF], lo[NF];
#pragma unroll
    for (int q = 0; q < NF; ++q) {
        hi[q] = 0ull;
        lo[q] = ~0ull;
    }
    const long long n2 = n >> 1;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n2;
         t += (long long)gridDim.x * blockDim.x) {
#pragma unroll
        for (int q = 0; q < NF; ++q) {
            const double2 v = __ldg(reinterpret_cast<const double2 *>(p.f[q]) + t);
            const unsigned long long k0 = fx_key((unsigned long long)__double_as_longlong(v.x));
            const unsigned long long k1 = fx_key((unsigned long long)__double_as_longlong(v.y));
            const unsigned long long kh = k0 > k1 ? k0 : k1, kl = k0 > k1 ? k1 : k0;
            hi[q] = kh > hi[q] ? kh : hi[q];
            lo[q] = kl < lo[q] ? kl : lo[q];
        }
    }
    if ((n & 1) && blockIdx.x == 0 && threadIdx.x == 0) {
#pragma unroll
        for (int q = 0; q < NF; ++q) {
            const unsigned long long k =
                fx_key((unsigned long long)__double_as_longlong(p.f[q][n - 1]));
            hi[q] = k > hi[q] ? k : hi[q];
            lo[q] = k < lo[q] ? k : lo[q];
        }
    }
    __shared__ unsigned long long red[2 * NF];
    if (threadIdx.x < NF) {
        red[threadIdx.x] = 0ull;
        red[NF + threadIdx.x] = ~0ull;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NF; ++q) {
        unsigned long long a = hi[q], b = lo[q];
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long x = __shfl_xor_sync(0xffffffffu, a, o);
            const unsigned long long y = __shfl_xor_sync(0xffffffffu, b, o);
            a = x > a ? x : a;
            b = y < b ? y : b;
        }
        if ((threadIdx.x & 31) == 0) {
            atomicMax(&red[q], a);
            atomicMin(&red[NF + q], b);
        }
    }
    __syncthreads();
    if (threadIdx.x < NF)
        atomicMax(&stats[threadIdx.x], red[threadIdx.x]);
    else if (threadIdx.x < 2 * NF)
        atomicMin(&stats[threadIdx.x], red[threadIdx.x]);
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&stats[2 * NF], 1ull) == gridDim.x - 1;
    __syncthreads();
    if (!last || threadIdx.x >= 32) return;
    __threadfence();
    fx_plan(stats, plan, gamma_cp, gm1, form);
    if (threadIdx.x == 0) stats[2 * NF] = 0ull;
}

// F = round(f 2^s) - round(c 2^s) by integer operations on the binary64 bits, with
// the periodic halo if the copies have one; nothing to do in FX_PLAIN.  The copies are
// written in order, PER cells a thread (256 apart, so that a warp's stores and loads are
// contiguous; two where that still fills the chip), all loads ahead of the stores; the
// place in the box of a CTA's first cell is divided out once.  (A warp to each padded row
// instead left long rows to few warps, 2.7 ms for 65536 x 1 x 1, and narrow rows to few
// lanes.)
template <int PER>
__global__ void __launch_bounds__(256) fx_quantize_kernel(FxPtrs p, Geom g, const FxPlan *plan) {
    if (plan->kern == FX_PLAIN) return;
    int s[NF], zero[NF];
    unsigned long long C[NF];
#pragma unroll
    for (int q = 0; q < NF; ++q) {
        s[q] = plan->s[q];
        zero[q] = plan->zero[q];
        C[q] = plan->C[q];
    }
    auto fix = [&](double v, int q) -> long long {
        return zero[q] ? 0ll
                       : (long long)(fx_round_grid((unsigned long long)__double_as_longlong(v), s[q]) -
                                     C[q]);
    };
    const unsigned px = p.g.px, py = p.py;
    for (long long t0 = blockIdx.x * (256ll * PER); t0 < p.g.elems; t0 += gridDim.x * (256ll * PER)) {
        const unsigned row0 = (unsigned)(t0 >> 32 ? t0 / px : (unsigned)t0 / px);
        const unsigned x0 = (unsigned)t0 - row0 * px;
        const unsigned k0 = row0 / py, j0 = row0 - k0 * py;
        long long src[PER];
        double v[PER][NF];
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            // the cell of the state that this cell of the copies holds
            const bool in = t0 + threadIdx.x + 256 * u < p.g.elems;
            const unsigned x = x0 + (in ? threadIdx.x + 256 * u : 0u), rows = x / px;
            const unsigned j = j0 + rows, planes = j / py;
            src[u] = wrap_near((int)(k0 + planes) - p.halo, g.nz) * g.pxy +
                     (long long)wrap_near((int)(j - planes * py) - p.halo, g.ny) * g.px +
                     wrap_near((int)(x - rows * px) - p.halo, g.nx);
        }
#pragma unroll
        for (int q = 0; q < NF; ++q)
#pragma unroll
            for (int u = 0; u < PER; ++u) v[u][q] = __ldg(p.f[q] + src[u]);
#pragma unroll
        for (int q = 0; q < NF; ++q)
#pragma unroll
            for (int u = 0; u < PER; ++u)
                if (t0 + threadIdx.x + 256 * u < p.g.elems)
                    p.F[q][t0 + threadIdx.x + 256 * u] = fix(v[u][q], q);
    }
}

// ---- integer stencil numerators (Eq. 13 points, sixth order) ---------------

// 45 (F1 - F-1) - 9 (F2 - F-2) + (F3 - F-3): first derivative x 60 dx.
template <int AX, class V>
__device__ __forceinline__ long long nd1(const V &F) {
    constexpr int ox = AX == 0, oy = AX == 1, oz = AX == 2;
    const long long a1 = F(ox, oy, oz) - F(-ox, -oy, -oz);
    const long long a2 = F(2 * ox, 2 * oy, 2 * oz) - F(-2 * ox, -2 * oy, -2 * oz);
    const long long a3 = F(3 * ox, 3 * oy, 3 * oz) - F(-3 * ox, -3 * oy, -3 * oz);
    return 45 * a1 - 9 * a2 + a3;
}

// -490 F0 + 270 (F1 + F-1) - 27 (F2 + F-2) + 2 (F3 + F-3): second derivative x 180 dx^2.
template <int AX, class V>
__device__ __forceinline__ long long nd2(const V &F, long long F0) {
    constexpr int ox = AX == 0, oy = AX == 1, oz = AX == 2;
    const long long s1 = F(ox, oy, oz) + F(-ox, -oy, -oz);
    const long long s2 = F(2 * ox, 2 * oy, 2 * oz) + F(-2 * ox, -2 * oy, -2 * oz);
    const long long s3 = F(3 * ox, 3 * oy, 3 * oz) + F(-3 * ox, -3 * oy, -3 * oz);
    return -490 * F0 + 270 * s1 - 27 * s2 + 2 * s3;
}

// 270 S1 - 27 S2 + 2 S3 over the face diagonals: mixed derivative x 720 dx^2.
template <int A, int B, class V>
__device__ __forceinline__ long long ndab(const V &F) {
    constexpr int ax = A == 0, ay = A == 1, az = A == 2;
    constexpr int bx = B == 0, by = B == 1, bz = B == 2;
    long long S[3];
#pragma unroll
    for (int m = 1; m <= 3; ++m) {
        const long long pp = F(m * (ax + bx), m * (ay + by), m * (az + bz));
        const long long mm = F(-m * (ax + bx), -m * (ay + by), -m * (az + bz));
        const long long pm = F(m * (ax - bx), m * (ay - by), m * (az - bz));
        const long long mp = F(-m * (ax - bx), -m * (ay - by), -m * (az - bz));
        S[m - 1] = (pp + mm) - (pm + mp);
    }
    return 270 * S[0] - 27 * S[1] + 2 * S[2];
}

// (double)N 2^k exactly for the integer numerator N, by adding k to the
// exponent field of the converted value (k_hi = k << 20, the exponent's place in
// the high word); 0 stays 0.  Every product stays normal: 1 <= |N| < 2^63 and
// the plan keeps 2^-s within [2^-1010, 2^910].
__device__ __forceinline__ double fx_scaled(long long N, int k_hi) {
    const double v = (double)N;
    return N == 0 ? 0.0 : __hiloint2double(__double2hiint(v) + k_hi, __double2loint(v));
}

// Coefficients of the converted numerators (host side); the field scales
// 2^-s come from the device plan.  Every coefficient through which a
// term enters the right-hand side also carries the step dt (dts below; the host
// takes this path only for |dt| in [1e-100, 1e100], so that 1 / dt^2 stays in
// range).  The RHS so formed is dt times Eqs. B.1-B.4, and the RK update adds it
// to alpha w without multiplying it by dt.
struct FxCoefs {
    double c1dt;       // dts c1, c1 = 1 / (60 dx): first derivatives in the RHS and B = curl A
    double nu180;      // dts nu / (180 dx^2): nu lap u
    double nu2160;     // dts (nu + 3 zeta) / (2160 dx^2): (nu / 3 + zeta) grad(div u)
    double inv180dx2;  // 1 / (180 dx^2): lap A (in j, and times eta dts in Eq. B.4)
    double inv720dx2;  // 1 / (720 dx^2): grad(div A)
    double two_nu_c1sq;  // dts 2 nu c1^2: 2 nu S : S and 2 nu S grad ln rho from unscaled gradients
    double K_c1sq;       // dts K c1^2: K |grad xi|^2 (conduction)
    double zeta_c1sq;    // dts zeta c1^2: zeta (div u)^2
    double eta_dt;       // dts eta
    double hc_dt;        // dts (H - C)
    double K_dt;         // dts K
    double amp_dt[3];    // dts times the forcing amplitudes
    double inv_dt2;      // 1 / dts^2: |B|^2 of the CFL speed from the dts-scaled B
    // FX_GROUP:
    double sg;         // two_nu_c1sq 4/3: 2 nu S . grad ln rho from X = 3/4 S
    double s2;         // two_nu_c1sq 16/9 / T_ref: 2 nu S : S / T
    double jb;         // -c1dt / (720 dx^2): j x B / rho from -j and B
    double j2;         // eta_dt / (720 dx^2)^2 / T_ref: eta j^2 / (rho T)
    double eta180;     // eta_dt / (180 dx^2): eta lap A
    double c1sq;       // 1 / (60 dx)^2
    double inv_T_ref;  // c_p (gamma - 1) / cs2_ref
    float c1f, cs2_ref_f;  // c1 and cs2_ref rounded up (the CFL bound)
    // unequal spacing (dx above then stands for the smallest, h): the numerators of axis
    // a times h / dx_a, (h / dx_a)^2 and, for the planes xy, xz, yz, h^2 / (dx_a dx_b),
    // each hi 2^-31 + lo 2^-62
    int r1h[3], r1l[3], r2h[3], r2l[3], rmh[3], rml[3];
};

// Eqs. B.1-B.4 at one cell as cell_physics computes them, times dts (the step
// folded into the coefficients of FxCoefs), with the gradients of ln rho, s and
// u passed without the grid factor c1 = 1 / (60 dx) (the integer stencil
// numerators after their field scale): every term is linear or quadratic in
// them, so c1 enters the coefficients (dts c1 for the advection terms inside
// their fused multiply-adds, dts c1 cs^2 for the pressure term, dts c1^2 in
// 2 nu, K and zeta) instead of 15 multiplications per cell on the FP64 pipe.
// B = curl A comes scaled by dts c1 (it meets c1 in three places, and dts
// reaches the Lorentz force and the induction through it).
template <bool EXT>
__device__ __forceinline__ void cell_physics_fx(const double (&u)[3], const double (&GL)[3],
                                                const double (&GS)[3], const double (&GU)[3][3],
                                                const double (&B)[3], const double (&viscl)[3],
                                                const double (&lapa)[3], const double (&J)[3],
                                                const DevCoefs<double> &k, const FxCoefs &fc,
                                                const double frc[3], double out[NF], double *cfl,
                                                double lapxi, const Thermo<double> &th) {
    const double c1 = fc.c1dt;
    const double rho_inv = th.rho_inv, cs2 = th.cs2, inv_T = th.inv_T;
    const double divR = GU[0][0] + GU[1][1] + GU[2][2];  // div u / c1
    const double third_div = divR * (1.0 / 3.0);
    // traceless rate of strain S / c1
    const double Sxx = GU[0][0] - third_div, Syy = GU[1][1] - third_div, Szz = GU[2][2] - third_div;
    const double Sxy = 0.5 * (GU[0][1] + GU[1][0]);
    const double Sxz = 0.5 * (GU[0][2] + GU[2][0]);
    const double Syz = 0.5 * (GU[1][2] + GU[2][1]);
    const double SS2 = Sxx * Sxx + Syy * Syy + Szz * Szz + 2.0 * (Sxy * Sxy + Sxz * Sxz + Syz * Syz);
    const double SG[3] = {Sxx * GL[0] + Sxy * GL[1] + Sxz * GL[2],
                          Sxy * GL[0] + Syy * GL[1] + Syz * GL[2],
                          Sxz * GL[0] + Syz * GL[1] + Szz * GL[2]};
    const double JxB[3] = {J[1] * B[2] - J[2] * B[1], J[2] * B[0] - J[0] * B[2],
                           J[0] * B[1] - J[1] * B[0]};
    const double UxB[3] = {u[1] * B[2] - u[2] * B[1], u[2] * B[0] - u[0] * B[2],
                           u[0] * B[1] - u[1] * B[0]};
    const double J2 = J[0] * J[0] + J[1] * J[1] + J[2] * J[2];
    // Eq. B.1
    out[0] = -(c1 * (u[0] * GL[0] + u[1] * GL[1] + u[2] * GL[2] + divR));
    // Eq. B.2
    const double c1cs2 = c1 * cs2;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        const double adv = u[0] * GU[m][0] + u[1] * GU[m][1] + u[2] * GU[m][2];
        const double press = c1cs2 * (GS[m] * k.inv_cp + GL[m]);
        const double visc = viscl[m] + fc.two_nu_c1sq * SG[m];
        out[1 + m] = fma(-c1, adv, visc) - press + JxB[m] * rho_inv + frc[m];
    }
    // Eq. B.3
    out[4] = fma(-c1, u[0] * GS[0] + u[1] * GS[1] + u[2] * GS[2],
                 (fc.eta_dt * J2 * rho_inv + fc.two_nu_c1sq * SS2) * inv_T);
    if (EXT) {
        double gxi2 = 0.0;  // |grad xi|^2 / c1^2
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const double gxi = k.gamma_cp * GS[m] + k.gm1 * GL[m];
            gxi2 += gxi * gxi;
        }
        out[4] += (fc.hc_dt * rho_inv + fc.zeta_c1sq * divR * divR) * inv_T +
                  rho_inv * (fc.K_dt * lapxi + fc.K_c1sq * gxi2);
    }
    // Eq. B.4
#pragma unroll
    for (int m = 0; m < 3; ++m) out[5 + m] = UxB[m] + fc.eta_dt * lapa[m];
    if (cfl) {
        const double b2 = (B[0] * B[0] + B[1] * B[1] + B[2] * B[2]) * fc.inv_dt2;
        const double u2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
        *cfl = sqrt(u2) + sqrt(cs2 + b2 * rho_inv);
    }
}

// One (x, y) column of the substep with integer stencils and binary64 products.  PF:
// per-field scales (FX_FIELD), so sums across the components of u or A are formed in
// binary64 from per-field integer numerators; otherwise one scale per group (the columns'
// FX_GROUP).
// IX addresses the int64 copies, with the halo or without.
template <bool PF, class IX, bool CFL, bool EXT>
__device__ __forceinline__ void fx_column(const SubstepArgs<double, double> &a, const FxPtrs &fx,
                                          const FxCoefs &fc, const FxPlan *plan,
                                          const double *etab, int i, int j, double &cfl) {
    // Each field's scale 2^-s is applied to its converted numerators
    // by an exponent add on the integer pipe (fx_scaled), so only the grid
    // coefficients -- kernel parameters, read from the constant bank -- multiply
    // on the FP64 pipe, and no scaled coefficient occupies registers (the
    // kernels sit at 255 registers).  In FX_GROUP the components of u and of A
    // share their exponent.
    int kh[NF];
#pragma unroll
    for (int q = 0; q < NF; ++q) kh[q] = -plan->s[q] * (1 << 20);
    // first derivative of field q from its numerator; the gradients of ln rho, s
    // and u stay without the factor c1 (cell_physics_fx applies it)
    auto d1 = [&](long long N, int q) -> double { return fx_scaled(N, kh[q]) * fc.c1dt; };
    auto d1r = [&](long long N, int q) -> double { return fx_scaled(N, kh[q]); };
    const int k0 = blockIdx.z * a.zchunk;
    const int k1 = min(k0 + a.zchunk, a.g.nz);
    IX ix;
    ix.set_xy(i, j, fx.g);
    double2 exy = make_double2(0.0, 0.0);
    if (a.force_on) {
        const double2 ex = a.ftab[i], ey = a.ftab[a.g.nx + j];
        exy.x = ex.x * ey.x - ex.y * ey.y;
        exy.y = ex.x * ey.y + ex.y * ey.x;
    }
    for (int kk = k0; kk < k1; ++kk) {
        ix.set_z(kk, fx.g);
        // (copies without a halo are addressed like the state)
        const long long o = std::is_same<IX, IdxPeriodic32>::value
                                ? ix(0, 0, 0)
                                : kk * a.g.pxy + (long long)j * a.g.px + i;
        // Centre values (the binary64 state) and the thermodynamic factors: at the
        // top of the cell in the CFL variant (substep 0), after the stencil sums in
        // the other; each placement measured fastest for its variant at 256^3
        // (8.30 against 8.78 ms, 7.89 against 8.64 ms), a matter of register
        // allocation at 255 registers.
        double lnrho = 0.0, ss = 0.0;
        Thermo<double> th;
        if constexpr (CFL) {
            lnrho = ldg(a.fin[0] + o);
            ss = ldg(a.fin[4] + o);
            th = thermo_factors<double>(lnrho, ss, a.k, etab);
        }
        double frc[3] = {0.0, 0.0, 0.0};
        if (a.force_on) {
            const double2 ez = a.ftab[a.g.nx + a.g.ny + kk];
            const double cph = exy.x * ez.x - exy.y * ez.y;
            frc[0] = fc.amp_dt[0] * cph;
            frc[1] = fc.amp_dt[1] * cph;
            frc[2] = fc.amp_dt[2] * cph;
        }
        using View = GlobalView<long long, IX>;
        const View Fl{fx.F[0], ix}, Fs{fx.F[4], ix};
        const View Fu[3] = {{fx.F[1], ix}, {fx.F[2], ix}, {fx.F[3], ix}};
        const View Fa[3] = {{fx.F[5], ix}, {fx.F[6], ix}, {fx.F[7], ix}};
        // first derivatives
        double gl[3], gs[3], gu[3][3], B[3];
        gl[0] = d1r(nd1<0>(Fl), 0);
        gl[1] = d1r(nd1<1>(Fl), 0);
        gl[2] = d1r(nd1<2>(Fl), 0);
        gs[0] = d1r(nd1<0>(Fs), 4);
        gs[1] = d1r(nd1<1>(Fs), 4);
        gs[2] = d1r(nd1<2>(Fs), 4);
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const int qu = PF ? 1 + m : 1;  // one live exponent in FX_GROUP
            gu[m][0] = d1r(nd1<0>(Fu[m]), qu);
            gu[m][1] = d1r(nd1<1>(Fu[m]), qu);
            gu[m][2] = d1r(nd1<2>(Fu[m]), qu);
        }
        if constexpr (PF) {
            B[0] = (fx_scaled(nd1<1>(Fa[2]), kh[7]) - fx_scaled(nd1<2>(Fa[1]), kh[6])) * fc.c1dt;
            B[1] = (fx_scaled(nd1<2>(Fa[0]), kh[5]) - fx_scaled(nd1<0>(Fa[2]), kh[7])) * fc.c1dt;
            B[2] = (fx_scaled(nd1<0>(Fa[1]), kh[6]) - fx_scaled(nd1<1>(Fa[0]), kh[5])) * fc.c1dt;
        } else {
            B[0] = d1(nd1<1>(Fa[2]) - nd1<2>(Fa[1]), 5);
            B[1] = d1(nd1<2>(Fa[0]) - nd1<0>(Fa[2]), 5);
            B[2] = d1(nd1<0>(Fa[1]) - nd1<1>(Fa[0]), 5);
        }
        // lap V_i = sum_a N2_aa(V_i) / (180 dx^2);
        // grad(div V)_i = [4 N2_ii(V_i) + NX_ij(V_j) + NX_ik(V_k)] / (720 dx^2);
        // component C of V contributes 4 N2_CC to entry C and its two mixed
        // numerators to the other two entries.
        double viscl[3], lapa[3], J[3];
        if constexpr (PF) {
            // per-field scaled numerators, summed across components in binary64
            double LU[3], GU[3], LA[3], GA[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int b1 = c == 0 ? 1 : 0, b2 = c == 2 ? 1 : 2;
                {
                    const long long c0 = Fu[c](0, 0, 0);
                    const long long xx = nd2<0>(Fu[c], c0), yy = nd2<1>(Fu[c], c0),
                                    zz = nd2<2>(Fu[c], c0);
                    const int k = kh[1 + c];
                    LU[c] = fx_scaled(xx + yy + zz, k);
                    const double own = fx_scaled(4 * (c == 0 ? xx : (c == 1 ? yy : zz)), k);
                    const double x1 = fx_scaled(c == 2 ? ndab<0, 2>(Fu[c]) : ndab<0, 1>(Fu[c]), k);
                    const double x2 = fx_scaled(c == 0 ? ndab<0, 2>(Fu[c]) : ndab<1, 2>(Fu[c]), k);
                    if (c == 0) {
                        GU[0] = own;
                        GU[1] = x1;
                        GU[2] = x2;
                    } else {
                        GU[c] += own;
                        GU[b1] += x1;
                        GU[b2] += x2;
                    }
                }
                {
                    const long long c0 = Fa[c](0, 0, 0);
                    const long long xx = nd2<0>(Fa[c], c0), yy = nd2<1>(Fa[c], c0),
                                    zz = nd2<2>(Fa[c], c0);
                    const int k = kh[5 + c];
                    LA[c] = fx_scaled(xx + yy + zz, k);
                    const double own = fx_scaled(4 * (c == 0 ? xx : (c == 1 ? yy : zz)), k);
                    const double x1 = fx_scaled(c == 2 ? ndab<0, 2>(Fa[c]) : ndab<0, 1>(Fa[c]), k);
                    const double x2 = fx_scaled(c == 0 ? ndab<0, 2>(Fa[c]) : ndab<1, 2>(Fa[c]), k);
                    if (c == 0) {
                        GA[0] = own;
                        GA[1] = x1;
                        GA[2] = x2;
                    } else {
                        GA[c] += own;
                        GA[b1] += x1;
                        GA[b2] += x2;
                    }
                }
            }
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                viscl[m] = fma(LU[m], fc.nu180, GU[m] * fc.nu2160);
                lapa[m] = LA[m] * fc.inv180dx2;
                J[m] = fma(GA[m], fc.inv720dx2, -lapa[m]);
            }
        } else {
            long long LU[3], GU[3];
            {
                const long long c0 = Fu[0](0, 0, 0);
                const long long xx = nd2<0>(Fu[0], c0), yy = nd2<1>(Fu[0], c0), zz = nd2<2>(Fu[0], c0);
                LU[0] = xx + yy + zz;
                GU[0] = 4 * xx;
                GU[1] = ndab<0, 1>(Fu[0]);
                GU[2] = ndab<0, 2>(Fu[0]);
            }
            {
                const long long c0 = Fu[1](0, 0, 0);
                const long long xx = nd2<0>(Fu[1], c0), yy = nd2<1>(Fu[1], c0), zz = nd2<2>(Fu[1], c0);
                LU[1] = xx + yy + zz;
                GU[1] += 4 * yy;
                GU[0] += ndab<0, 1>(Fu[1]);
                GU[2] += ndab<1, 2>(Fu[1]);
            }
            {
                const long long c0 = Fu[2](0, 0, 0);
                const long long xx = nd2<0>(Fu[2], c0), yy = nd2<1>(Fu[2], c0), zz = nd2<2>(Fu[2], c0);
                LU[2] = xx + yy + zz;
                GU[2] += 4 * zz;
                GU[0] += ndab<0, 2>(Fu[2]);
                GU[1] += ndab<1, 2>(Fu[2]);
            }
            // the same two sums for A; j = grad(div A) - lap A
            long long LA[3], GA[3];
            {
                const long long c0 = Fa[0](0, 0, 0);
                const long long xx = nd2<0>(Fa[0], c0), yy = nd2<1>(Fa[0], c0), zz = nd2<2>(Fa[0], c0);
                LA[0] = xx + yy + zz;
                GA[0] = 4 * xx;
                GA[1] = ndab<0, 1>(Fa[0]);
                GA[2] = ndab<0, 2>(Fa[0]);
            }
            {
                const long long c0 = Fa[1](0, 0, 0);
                const long long xx = nd2<0>(Fa[1], c0), yy = nd2<1>(Fa[1], c0), zz = nd2<2>(Fa[1], c0);
                LA[1] = xx + yy + zz;
                GA[1] += 4 * yy;
                GA[0] += ndab<0, 1>(Fa[1]);
                GA[2] += ndab<1, 2>(Fa[1]);
            }
            {
                const long long c0 = Fa[2](0, 0, 0);
                const long long xx = nd2<0>(Fa[2], c0), yy = nd2<1>(Fa[2], c0), zz = nd2<2>(Fa[2], c0);
                LA[2] = xx + yy + zz;
                GA[2] += 4 * zz;
                GA[0] += ndab<0, 2>(Fa[2]);
                GA[1] += ndab<1, 2>(Fa[2]);
            }
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                viscl[m] = fma(fx_scaled(LU[m], kh[1]), fc.nu180, fx_scaled(GU[m], kh[1]) * fc.nu2160);
                lapa[m] = fx_scaled(LA[m], kh[5]) * fc.inv180dx2;
                J[m] = fma(fx_scaled(GA[m], kh[5]), fc.inv720dx2, -lapa[m]);
            }
        }
        // EXT: lap xi = gamma / c_p lap s + (gamma - 1) lap ln rho (conduction)
        double lapxi = 0.0;
        if (EXT) {
            const long long l0 = Fl(0, 0, 0), s0 = Fs(0, 0, 0);
            const long long LL = nd2<0>(Fl, l0) + nd2<1>(Fl, l0) + nd2<2>(Fl, l0);
            const long long LS = nd2<0>(Fs, s0) + nd2<1>(Fs, s0) + nd2<2>(Fs, s0);
            lapxi = a.k.gamma_cp * (fx_scaled(LS, kh[4]) * fc.inv180dx2) +
                    a.k.gm1 * (fx_scaled(LL, kh[0]) * fc.inv180dx2);
        }
        if constexpr (!CFL) {
            lnrho = ldg(a.fin[0] + o);
            ss = ldg(a.fin[4] + o);
            th = thermo_factors<double>(lnrho, ss, a.k, etab);
        }
        const double u[3] = {ldg(a.fin[1] + o), ldg(a.fin[2] + o), ldg(a.fin[3] + o)};
        double rhs[NF];
        if (CFL) {
            double v;
            cell_physics_fx<EXT>(u, gl, gs, gu, B, viscl, lapa, J, a.k, fc, frc, rhs, &v, lapxi, th);
            cfl = (v > cfl || v != v) ? v : cfl;
        } else {
            cell_physics_fx<EXT>(u, gl, gs, gu, B, viscl, lapa, J, a.k, fc, frc, rhs, nullptr, lapxi,
                                 th);
        }
        // the RK update of rk_update, the RHS already multiplied by dt
#pragma unroll
        for (int q = 0; q < NF; ++q) {
            double wn = rhs[q];
            if (!a.s0) wn = a.alpha * a.w[q][o] + wn;
            a.w[q][o] = wn;
            a.fout[q][o] = ldg(a.fin[q] + o) + a.beta * wn;
        }
    }
}

// How a form's int64 copies are addressed.
template <int FORM> struct FxIndex { using type = IdxPadded; };
template <> struct FxIndex<FX_COLUMNS> { using type = IdxPeriodic32; };

// ---- FX_GROUP: integer stencils, integer products --------------------------------
//
// A CTA owns a 16 x 16 column tile and marches along z with two threads per cell:
// eight warps take the equations of ln rho, u and s, eight warps A, the pressure and
// the thermodynamic factors (4 warps per scheduler at 128 registers).  A ring of seven
// planes in shared memory holds the tile with its halo (22 x 22 cells x eight fields,
// 31 KB a plane, 217 KB: one CTA per SM), each plane fetched by one TMA box.  There is
// no eighth slot to prefetch into: a cell's stencils are all taken first, and plane
// z + 4 lands in plane z - 3's slot while the products, conversions and the
// Runge-Kutta update of plane z run.
// Measured at 256^3, ms per substep (s = 1, 2): 7.35 with binary64 products (bound by
// the FP64 pipe, 179 instructions a cell); these integer products with stencil points
// loaded through L1 5.95 (load latency at 2 warps per scheduler); one thread per cell
// on the ring 3.72; two threads in lockstep between CTA barriers 4.11; without CTA
// barriers (FxMarch) 3.40; with the halves balanced 3.18, and 3.29 since conversions take
// every size and the pressure's gradients a scale each.  Bound now by the issue of its
// 4270 instructions a cell (about half the issue slots; ALU 48%, FP64 pipe 55%).
constexpr int FXT = 16;                            // tile edge
constexpr int FXR = FXT + 2 * R;                   // staged row
constexpr int FX_FIELD_TILE = FXR * FXR;           // cells of one staged field plane
constexpr int FX_PLANE = NF * FX_FIELD_TILE;       // int64 of one ring slot
constexpr int FX_SLOTS = 2 * R + 1;
constexpr unsigned FX_PLANE_BYTES = FX_PLANE * 8;
constexpr int FX_WARPS = 2 * FXT * FXT / 32;
constexpr int FX_XCH = 6;                          // doubles a cell's A thread hands to its u thread
constexpr size_t FX_SMEM =
    (size_t)FX_SLOTS * FX_PLANE_BYTES + 8 * (256 + FX_XCH * FXT * FXT);

__device__ __forceinline__ unsigned fx_smem_u32(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
// A load that stays where it is written (the compiler would sink it to its use).
__device__ __forceinline__ double fx_load_now(const double *p) {
    double v;
    asm volatile("ld.global.f64 %0, [%1];\n" : "=d"(v) : "l"(p));
    return v;
}
// Whether the phase of `bar` with the given parity has completed (a poll that does not
// find it so returns after about 3.8 us).
__device__ __forceinline__ bool fx_poll(fx_u64 *bar, unsigned parity) {
    unsigned done;
    asm volatile(
        "{\n .reg .pred p;\n"
        " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(fx_smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0;
}
// Wait for it; false after `polls` polls.
__device__ __forceinline__ bool fx_wait(fx_u64 *bar, unsigned parity, unsigned polls) {
    for (unsigned it = 0; it < polls; ++it)
        if (fx_poll(bar, parity)) return true;
    return false;
}
// One plane (padded plane index pz) of the tile whose first staged cell is (x, y).
__device__ __forceinline__ void fx_fetch(long long *dst, const CUtensorMap *map, fx_u64 *bar, int x,
                                         int y, int pz) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(fx_smem_u32(bar)),
                 "r"(FX_PLANE_BYTES)
                 : "memory");
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%3, %4, %5, %6}], [%2];\n" ::"r"(fx_smem_u32(dst)),
        "l"(reinterpret_cast<fx_u64>(map)), "r"(fx_smem_u32(bar)), "r"(x), "r"(y), "r"(pz), "r"(0)
        : "memory");
}

// One field around a thread's cell in the ring: `c` its centre in slot 0, slot[d]
// the offset of plane z - 3 + d.
struct FxView {
    const long long *c;
    const int (&slot)[FX_SLOTS];
    __device__ __forceinline__ long long operator()(int dx, int dy, int dz) const {
        return c[slot[dz + R] + dy * FXR + dx];
    }
};

// One axis of a field: first-derivative numerator d (x 60 dx) and the sums s1 = F1 +
// F-1, n2 = -(F2 + F-2), s3 = F3 + F-3 of the second derivative (every weight below
// is then positive, as fx_wmac wants).
struct FxAxis {
    long long d, s1, n2, s3;
};
template <int AX>
__device__ __forceinline__ FxAxis fx_axis(const FxView &F) {
    constexpr int ox = AX == 0, oy = AX == 1, oz = AX == 2;
    const long long p1 = F(ox, oy, oz), m1 = F(-ox, -oy, -oz);
    const long long p2 = F(2 * ox, 2 * oy, 2 * oz), m2 = F(-2 * ox, -2 * oy, -2 * oz);
    const long long p3 = F(3 * ox, 3 * oy, 3 * oz), m3 = F(-3 * ox, -3 * oy, -3 * oz);
    FxAxis a;
    a.d = 45 * (p1 - m1) + 9 * (m2 - p2) + (p3 - m3);
    a.s1 = p1 + m1;
    a.n2 = -p2 - m2;
    a.s3 = p3 + m3;
    return a;
}

// v += N_AB (NEG: v -= N_AB), N_AB the mixed-derivative numerator 270 S1 - 27 S2 +
// 2 S3 (x 720 dx^2).
template <int A, int B, bool NEG>
__device__ __forceinline__ void fx_mixed(const FxView &F, FxWide &v) {
    constexpr int ax = A == 0, ay = A == 1, az = A == 2;
    constexpr int bx = B == 0, by = B == 1, bz = B == 2;
    constexpr int W[3] = {270, 27, 2};
#pragma unroll
    for (int m = 1; m <= 3; ++m) {
        const long long pp = F(m * (ax + bx), m * (ay + by), m * (az + bz));
        const long long mm = F(-m * (ax + bx), -m * (ay + by), -m * (az + bz));
        const long long pm = F(m * (ax - bx), m * (ay - by), m * (az - bz));
        const long long mp = F(-m * (ax - bx), -m * (ay - by), -m * (az - bz));
        const bool minus = NEG != (m == 2);
        fx_wmac(v, minus ? (pm + mp) - (pp + mm) : (pp + mm) - (pm + mp), W[m - 1]);
    }
}

// lap F (x 180 dx^2) from its three axes and the centre.
__device__ __forceinline__ FxWide fx_lap(const FxAxis (&a)[3], long long f0) {
    FxWide w = {0, 0};
    fx_wmac(w, -f0, 1470);
    fx_wmac(w, a[0].s1 + a[1].s1 + a[2].s1, 270);
    fx_wmac(w, a[0].n2 + a[1].n2 + a[2].n2, 27);
    fx_wmac(w, a[0].s3 + a[1].s3 + a[2].s3, 2);
    return w;
}

// Unequal spacing: each numerator is brought to the smallest spacing's factor by one
// fixed-point product, then sums run in 64 bits: first derivatives in the units above,
// second ones over 2^6 (a quantum of 64 beside the 180 that the rounding of F leaves
// in a second-derivative numerator), mixed ones and grad(div) over 2^8.
template <bool ANISO>
__device__ __forceinline__ long long fx_first(long long d, const FxCoefs &fc, int a) {
    return ANISO ? fx_mulfrac(d, fc.r1h[a], fc.r1l[a]) : d;
}
__device__ __forceinline__ long long fx_second(const FxAxis &a, long long f0, const FxCoefs &fc, int ax) {
    FxWide w = {0, 0};
    fx_wmac(w, -f0, 490);
    fx_wmac(w, a.s1, 270);
    fx_wmac(w, a.n2, 27);
    fx_wmac(w, a.s3, 2);
    return fx_mulfrac(fx_shift96<6>(fx_wide96(w)), fc.r2h[ax], fc.r2l[ax]);
}
template <int A, int B, bool NEG>
__device__ __forceinline__ long long fx_mixed_scaled(const FxView &F, const FxCoefs &fc) {
    FxWide w = {0, 0};
    fx_mixed<A, B, NEG>(F, w);
    constexpr int pl = Plane<A, B>::id;
    return fx_mulfrac(fx_shift96<6>(fx_wide96(w)), fc.rmh[pl], fc.rml[pl]) >> 2;
}
template <int C>
__device__ __forceinline__ void fx_u_component_scaled(const FxView &F, long long f0, const FxCoefs &fc,
                                                      long long (&GD)[3], long long (&G)[3],
                                                      long long &LU) {
    constexpr int B1 = C == 0 ? 1 : 0, B2 = C == 2 ? 1 : 2;
    const FxAxis u[3] = {fx_axis<0>(F), fx_axis<1>(F), fx_axis<2>(F)};
    long long n[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        G[a] = fx_first<true>(u[a].d >> 2, fc, a);
        n[a] = fx_second(u[a], f0, fc, a);
    }
    LU = n[0] + n[1] + n[2];
    GD[C] += n[C];
    GD[B1] += fx_mixed_scaled<(C < B1 ? C : B1), (C < B1 ? B1 : C), false>(F, fc);
    GD[B2] += fx_mixed_scaled<(C < B2 ? C : B2), (C < B2 ? B2 : C), false>(F, fc);
}
template <int C>
__device__ __forceinline__ void fx_a_component_scaled(const FxView &F, long long f0, const FxCoefs &fc,
                                                      long long (&Jn)[3], long long (&B)[3],
                                                      long long &LA) {
    constexpr int B1 = C == 0 ? 1 : 0, B2 = C == 2 ? 1 : 2;
    const FxAxis v[3] = {fx_axis<0>(F), fx_axis<1>(F), fx_axis<2>(F)};
    if (C == 0) {
        B[2] -= fx_first<true>(v[1].d >> 3, fc, 1);
        B[1] += fx_first<true>(v[2].d >> 3, fc, 2);
    } else if (C == 1) {
        B[2] += fx_first<true>(v[0].d >> 3, fc, 0);
        B[0] -= fx_first<true>(v[2].d >> 3, fc, 2);
    } else {
        B[1] -= fx_first<true>(v[0].d >> 3, fc, 0);
        B[0] += fx_first<true>(v[1].d >> 3, fc, 1);
    }
    const long long n[3] = {fx_second(v[0], f0, fc, 0), fx_second(v[1], f0, fc, 1),
                            fx_second(v[2], f0, fc, 2)};
    LA = n[0] + n[1] + n[2];
    Jn[C] += n[B1] + n[B2];
    Jn[B1] += fx_mixed_scaled<(C < B1 ? C : B1), (C < B1 ? B1 : C), true>(F, fc);
    Jn[B2] += fx_mixed_scaled<(C < B2 ? C : B2), (C < B2 ? B2 : C), true>(F, fc);
}

// Component C of u: G[a] = d_a u_C (x 60 dx, over 4); its share of V, the viscous
// numerators 12 lap u + grad(div u) (x 2160 dx^2; with EXT, for any zeta, grad(div u)
// alone, x 720 dx^2, and LU = lap u_C).
template <int C, bool EXT>
__device__ __forceinline__ void fx_u_component(const FxView &F, long long f0, FxWide (&V)[3],
                                               long long (&G)[3], FxWide &LU) {
    constexpr int B1 = C == 0 ? 1 : 0, B2 = C == 2 ? 1 : 2;
    const FxAxis u[3] = {fx_axis<0>(F), fx_axis<1>(F), fx_axis<2>(F)};
#pragma unroll
    for (int a = 0; a < 3; ++a) G[a] = u[a].d >> 2;
    if (EXT) {
        fx_wmac(V[C], -f0, 1960);
        fx_wmac(V[C], u[C].s1, 1080);
        fx_wmac(V[C], u[C].n2, 108);
        fx_wmac(V[C], u[C].s3, 8);
        LU = fx_lap(u, f0);
    } else {
        fx_wmac(V[C], -f0, 19600);
        fx_wmac(V[C], u[C].s1, 4320);
        fx_wmac(V[C], u[C].n2, 432);
        fx_wmac(V[C], u[C].s3, 32);
        fx_wmac(V[C], u[B1].s1 + u[B2].s1, 3240);
        fx_wmac(V[C], u[B1].n2 + u[B2].n2, 324);
        fx_wmac(V[C], u[B1].s3 + u[B2].s3, 24);
    }
    fx_mixed<(C < B1 ? C : B1), (C < B1 ? B1 : C), false>(F, V[B1]);
    fx_mixed<(C < B2 ? C : B2), (C < B2 ? B2 : C), false>(F, V[B2]);
}

// Component C of A: its share of B = curl A (x 60 dx, over 8) and of Jn = 4 (lap A -
// grad(div A)) (x 720 dx^2, minus the current); LA = lap A_C (x 180 dx^2).
template <int C>
__device__ __forceinline__ void fx_a_component(const FxView &F, long long f0, FxWide (&Jn)[3],
                                               long long (&B)[3], FxWide &LA) {
    constexpr int B1 = C == 0 ? 1 : 0, B2 = C == 2 ? 1 : 2;
    const FxAxis v[3] = {fx_axis<0>(F), fx_axis<1>(F), fx_axis<2>(F)};
    if (C == 0) {
        B[2] -= v[1].d >> 3;
        B[1] += v[2].d >> 3;
    } else if (C == 1) {
        B[2] += v[0].d >> 3;
        B[0] -= v[2].d >> 3;
    } else {
        B[1] -= v[0].d >> 3;
        B[0] += v[1].d >> 3;
    }
    LA = fx_lap(v, f0);
    fx_wmac(Jn[C], -f0, 3920);
    fx_wmac(Jn[C], v[B1].s1 + v[B2].s1, 1080);
    fx_wmac(Jn[C], v[B1].n2 + v[B2].n2, 108);
    fx_wmac(Jn[C], v[B1].s3 + v[B2].s3, 8);
    fx_mixed<(C < B1 ? C : B1), (C < B1 ? B1 : C), true>(F, Jn[B1]);
    fx_mixed<(C < B2 ? C : B2), (C < B2 ? B2 : C), true>(F, Jn[B2]);
}

// An upper bound of a positive double as binary32 (its exponent within binary32's).
__device__ __forceinline__ float fx_float_up(double v) {
    const long long b = __double_as_longlong(v);
    return __int_as_float((int)((b - (896ll << 52)) >> 29) + 1);
}

// The Runge-Kutta update of rk_update, the RHS already multiplied by dt.
__device__ __forceinline__ void fx_update(const SubstepArgs<double, double> &a, bool active, int q,
                                          long long o, double f, double w, double rhs) {
    double wn = rhs;
    if (!a.s0) wn = a.alpha * w + wn;
    if (active) {
        a.w[q][o] = wn;
        a.fout[q][o] = f + a.beta * wn;
    }
}

__device__ __forceinline__ void fx_arrive(fx_u64 *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(fx_smem_u32(bar)) : "memory");
}

// What a CTA's warps share in the march along z.  No barrier spans the CTA inside the
// march: a warp waits for the plane it needs, and the last of the sixteen to finish
// its stencils of plane z asks for plane z + 4, so that some warps' stencils (shared
// memory, integer pipes) run beside others' products and updates (FP64 pipe).
struct FxShared {
    fx_u64 full[FX_SLOTS];           // a plane has landed
    fx_u64 given[FX_WARPS / 2];      // the A warp's exchange values are written ...
    fx_u64 taken[FX_WARPS / 2];      // ... and read by the u warp of the same cells
    unsigned done;                   // warps that have finished their stencils (cumulative)
    unsigned polls;                  // of a wait before it gives up
    unsigned fetched;                // planes asked for, plane n of them into slot n % FX_SLOTS
    int cfl_low;                     // the CTA's cfl_low below (bits of a positive float)
};
struct FxMarch {
    const CUtensorMap *map;
    long long *sm;
    FxShared *sh;
    int x0, y0, z0, z1;
    int slot[FX_SLOTS];  // ring offsets of planes z-3 .. z+3, rolled by one per plane
    int last;            // the slot that plane z + 3 is in, and the parity of its fill
    unsigned parity;
    bool ok;             // false once a bounded wait has run out
    // wait in the march: the limit is only read where the first poll finds nothing
    __device__ __forceinline__ bool wait(fx_u64 *bar, unsigned p) {
        return fx_poll(bar, p) || fx_wait(bar, p, *(volatile unsigned *)&sh->polls);
    }
    // plane z + 3 has landed
    __device__ __forceinline__ bool arrive() {
        ok = __all_sync(0xffffffffu, wait(&sh->full[last], parity));
        return ok;
    }
    // this warp has taken its stencils of plane z; once all have, plane z - 3's slot
    // is free for plane z + 4
    __device__ __forceinline__ void refill(int z) {
        __syncwarp();
        if ((threadIdx.x & 15) == 0 && (threadIdx.y & 1) == 0) {
            __threadfence_block();
            const unsigned n = atomicAdd(&sh->done, 1u) + 1u;
            if (n == FX_WARPS * (unsigned)(z - z0 + 1) && z + 1 < z1) {
                __threadfence_block();
                atomicAdd(&sh->fetched, 1u);
                fx_fetch(sm + slot[0], map, &sh->full[last == FX_SLOTS - 1 ? 0 : last + 1], x0, y0,
                         z + 7);
            }
        }
    }
    __device__ __forceinline__ void next() {
        const int first = slot[0];
#pragma unroll
        for (int d = 0; d < FX_SLOTS - 1; ++d) slot[d] = slot[d + 1];
        slot[FX_SLOTS - 1] = first;
        parity ^= last == FX_SLOTS - 1;
        last = last == FX_SLOTS - 1 ? 0 : last + 1;
    }
};

// Units of both halves: with kl, ku, ks, ka the binary exponents -s of the scales of
// ln rho, u, s and A, a stencil numerator N stands for N 2^k; GL, GS, GU carry
// 2^(k+2), B 2^(ka+3), J 2^(ka+9), X = 3/4 S 2^(ku+2), each below 2^60.8 as fx_split
// wants.

// The A half: A and the gradients of ln rho and s; dA/dt, the CFL speed, and for the
// cell's other thread (through xch) the pressure and Lorentz forces, the advection
// and conduction of s, eta j^2 / rho and 1/T.  (Which half takes which term is a
// matter of balance: with the pressure and the entropy's advection in the u half,
// that half ran 17.6 and this one 13.3 thousand cycles a plane.)
template <bool CFL, bool EXT, bool ANISO>
__device__ __forceinline__ void fx_march_a(const SubstepArgs<double, double> &a, const FxCoefs &fc,
                                           const FxPlan *plan, const fx_u64 *etab, double *xch,
                                           FxMarch &m, int i, int j, double &cfl) {
    const bool active = i < a.g.nx && j < a.g.ny;
    const int kl = -plan->s[0], ku = -plan->s[1], ks = -plan->s[4], ka = -plan->s[5];
    const long long Cu[3] = {(long long)plan->C[1], (long long)plan->C[2], (long long)plan->C[3]};
    const double c1cs2_ref = fc.c1dt * a.k.cs2_ref;
    // sh->cfl_low: the largest CFL speed known so far, rounded down (the CTA's own and,
    // from the start, what other CTAs have reported); cells whose upper bound lies below
    // it need no exact speed (two square roots: 1150 FP64-pipe cycles)
    const long long *const ring = m.sm + (threadIdx.y + R) * FXR + threadIdx.x + R;
    fx_u64 *const given = &m.sh->given[threadIdx.y >> 1], *const taken = &m.sh->taken[threadIdx.y >> 1];
    const int z0 = m.z0;
    for (int z = z0; z < m.z1; ++z) {
        if (!m.arrive()) break;
        const long long o =
            AC_BC(z * a.g.pxy + (long long)j * a.g.px + i, active ? a.g.elems : 1ll << 62, AC_BC_TILE_OUT);
        // the cell's own values: asked for ahead of the stencils, needed after them
        double f0[3] = {}, w0[3] = {}, lnrho = 0.0, ss = 0.0;
        if (active) {
            lnrho = fx_load_now(a.fin[0] + o);
            ss = fx_load_now(a.fin[4] + o);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                f0[q] = fx_load_now(a.fin[5 + q] + o);
                if (!a.s0) w0[q] = fx_load_now(a.w[5 + q] + o);
            }
        }
        FxWide Jn[3] = {}, LA[3];
        long long Bn[3] = {0, 0, 0};
        const FxView Fx{ring + 5 * FX_FIELD_TILE, m.slot}, Fy{ring + 6 * FX_FIELD_TILE, m.slot},
            Fz{ring + 7 * FX_FIELD_TILE, m.slot};
        long long Js[3] = {0, 0, 0}, Ls[3];  // unequal spacing: -j over 2^8, lap A over 2^6
        if constexpr (ANISO) {
            fx_a_component_scaled<0>(Fx, Fx(0, 0, 0), fc, Js, Bn, Ls[0]);
            fx_a_component_scaled<1>(Fy, Fy(0, 0, 0), fc, Js, Bn, Ls[1]);
            fx_a_component_scaled<2>(Fz, Fz(0, 0, 0), fc, Js, Bn, Ls[2]);
        } else {
            fx_a_component<0>(Fx, Fx(0, 0, 0), Jn, Bn, LA[0]);
            fx_a_component<1>(Fy, Fy(0, 0, 0), Jn, Bn, LA[1]);
            fx_a_component<2>(Fz, Fz(0, 0, 0), Jn, Bn, LA[2]);
        }
        long long GL[3], GS[3];
        FxWide LL, LS;
        long long LLs = 0, LSs = 0;
        {
            const FxView Fl{ring, m.slot}, Fs{ring + 4 * FX_FIELD_TILE, m.slot};
            const FxAxis l[3] = {fx_axis<0>(Fl), fx_axis<1>(Fl), fx_axis<2>(Fl)};
            const FxAxis e[3] = {fx_axis<0>(Fs), fx_axis<1>(Fs), fx_axis<2>(Fs)};
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                GL[q] = fx_first<ANISO>(l[q].d >> 2, fc, q);
                GS[q] = fx_first<ANISO>(e[q].d >> 2, fc, q);
            }
            if (EXT && !ANISO) {
                LL = fx_lap(l, Fl(0, 0, 0));
                LS = fx_lap(e, Fs(0, 0, 0));
            }
            if (EXT && ANISO) {
                const long long l0 = Fl(0, 0, 0), e0 = Fs(0, 0, 0);
                LLs = fx_second(l[0], l0, fc, 0) + fx_second(l[1], l0, fc, 1) + fx_second(l[2], l0, fc, 2);
                LSs = fx_second(e[0], e0, fc, 0) + fx_second(e[1], e0, fc, 1) + fx_second(e[2], e0, fc, 2);
            }
        }
        FxSplit U[3];
#pragma unroll
        for (int q = 0; q < 3; ++q)
            U[q] = fx_split(ring[(1 + q) * FX_FIELD_TILE + m.slot[R]] + Cu[q]);
        m.refill(z);
        // (every thread of a ragged tile computes, the active ones load and store: the
        // barriers below want whole warps)
        FxSplit B[3], J[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            B[q] = fx_split(Bn[q]);
            J[q] = fx_split(ANISO ? Js[q] >> 1 : fx_shift96<9>(fx_wide96(Jn[q])));
        }
        // thermodynamic factors 1/rho, e^xi, e^-xi
        const double xi = a.k.gamma_cp * ss + a.k.gm1 * lnrho;
        const long long xx = fx_from_double55(xi);
        const double rho_inv = fx_exp55(-fx_from_double55(lnrho), etab, FX_L70);
        const double exi = fx_exp55(xx, etab, FX_L70), emxi = fx_exp55(-xx, etab, FX_L70);
        const double cjb = rho_inv * fc.jb, cp = exi * c1cs2_ref;
        // pressure and Lorentz force.  The two gradients are converted each with its own
        // scale: in a direction in which only the smaller-scaled field varies, a sum in the
        // other's units would keep only the bits left of those.
        const int ej = FX_EB + 44 + 2 * ka;
        double pl[3] = {cjb * fx_to_double(fx_det2(J[1], B[2], J[2], B[1]), ej),
                        cjb * fx_to_double(fx_det2(J[2], B[0], J[0], B[2]), ej),
                        cjb * fx_to_double(fx_det2(J[0], B[1], J[1], B[0]), ej)};
        FxSplit SS[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const double g = fma(a.k.inv_cp, fx_to_double(GS[q], FX_EB64 + 2 + ks),
                                 fx_to_double(GL[q], FX_EB64 + 2 + kl));
            pl[q] = fma(-cp, g, pl[q]);
            SS[q] = fx_split(GS[q]);
        }
        // entropy: advection, conduction, eta j^2 / rho
        double rs = -(fc.c1dt * fx_to_double(fx_dot3(U, SS), FX_EB + 34 + ku + ks));
        double h = fx_to_double(fx_dot3(J, J), FX_EB + 50 + 2 * ka) * (rho_inv * fc.j2);
        if (EXT) {
            h = fma(fc.inv_T_ref * fc.hc_dt, rho_inv, h);
            // lap xi and |grad xi|^2 / c1^2, xi = gamma s / c_p + (gamma - 1) ln rho
            const FxSplit SL[3] = {fx_split(GL[0]), fx_split(GL[1]), fx_split(GL[2])};
            const double ls = ANISO ? fx_to_double(LSs, FX_EB64 + 6 + ks)
                                    : fx_to_double(fx_wide96(LS), FX_EB + ks);
            const double ll = ANISO ? fx_to_double(LLs, FX_EB64 + 6 + kl)
                                    : fx_to_double(fx_wide96(LL), FX_EB + kl);
            const double lapxi = (a.k.gamma_cp * ls + a.k.gm1 * ll) * fc.inv180dx2;
            const double ss2 = fx_to_double(fx_dot3(SS, SS), FX_EB + 36 + 2 * ks);
            const double sl2 = fx_to_double(fx_dot3(SS, SL), FX_EB + 36 + ks + kl);
            const double ll2 = fx_to_double(fx_dot3(SL, SL), FX_EB + 36 + 2 * kl);
            const double gxi2 = a.k.gamma_cp * (a.k.gamma_cp * ss2 + 2.0 * a.k.gm1 * sl2) +
                                a.k.gm1 * a.k.gm1 * ll2;
            rs += rho_inv * (fc.K_dt * lapxi + fc.K_c1sq * gxi2);
        }
        // the u warp has read the values of the plane before
        if (z > z0) m.ok = __all_sync(0xffffffffu, m.wait(taken, (z - z0 - 1) & 1)) && m.ok;
#pragma unroll
        for (int q = 0; q < 3; ++q) xch[q * FXT * FXT] = pl[q];
        xch[3 * FXT * FXT] = h;
        xch[4 * FXT * FXT] = rs;
        xch[5 * FXT * FXT] = emxi;
        __syncwarp();
        if ((threadIdx.x & 15) == 0 && (threadIdx.y & 1) == 0) fx_arrive(given);
        const int eu = FX_EB + 35 + ku + ka;
        const double ub[3] = {fx_to_double(fx_det2(U[1], B[2], U[2], B[1]), eu),
                              fx_to_double(fx_det2(U[2], B[0], U[0], B[2]), eu),
                              fx_to_double(fx_det2(U[0], B[1], U[1], B[0]), eu)};
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const double la = ANISO ? fx_to_double(Ls[q], FX_EB64 + 6 + ka)
                                    : fx_to_double(fx_wide96(LA[q]), FX_EB + ka);
            fx_update(a, active, 5 + q, o, f0[q], w0[q], fma(fc.c1dt, ub[q], fc.eta180 * la));
        }
        if (CFL && active) {
            // upper bound of |u| + sqrt(c_s^2 + |B|^2 / rho) from the high words in
            // binary32; the exact speed only where that exceeds the largest known
            float u2 = 0.f, b2 = 0.f;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const float uf = fabsf((float)U[q].hi) + 1.f, bf = fabsf((float)B[q].hi) + 1.f;
                u2 = fmaf(uf, uf, u2);
                b2 = fmaf(bf, bf, b2);
            }
            // (floors: a scale that binary32 cannot hold only makes the bound larger)
            const float us = fmaxf(exp2f((float)(ku + 32)), 1e-37f),
                        bs = fmaxf(exp2f((float)(ka + 35)) * fc.c1f, 1e-18f);
            const float up =
                1.0001f * (us * sqrtf(u2) + sqrtf(fc.cs2_ref_f * fx_float_up(exi) +
                                                  bs * bs * b2 * fx_float_up(rho_inv)));
            if (!(up <= __int_as_float(*(volatile int *)&m.sh->cfl_low))) {
                const double x = ldg(a.fin[1] + o), y = ldg(a.fin[2] + o), zz = ldg(a.fin[3] + o);
                const double bb = fx_to_double(fx_dot3(B, B), FX_EB + 38 + 2 * ka) * fc.c1sq;
                const double c = sqrt(x * x + y * y + zz * zz) +
                                 sqrt(a.k.cs2_ref * exi + bb * rho_inv);
                if (c > cfl || c != c) {
                    cfl = c;
                    if (c < 1e30) atomicMax(&m.sh->cfl_low, __float_as_int(__double2float_rd(c)));
                }
            }
        }
        if (!m.ok) break;
        m.next();
    }
}

// The other half: the equations of ln rho, u and s.
template <bool EXT, bool ANISO>
__device__ __forceinline__ void fx_march_u(const SubstepArgs<double, double> &a, const FxCoefs &fc,
                                           const FxPlan *plan, const double *xch, FxMarch &m, int i, int j) {
    const bool active = i < a.g.nx && j < a.g.ny;
    const int kl = -plan->s[0], ku = -plan->s[1];
    const long long Cu[3] = {(long long)plan->C[1], (long long)plan->C[2], (long long)plan->C[3]};
    double2 exy = make_double2(0.0, 0.0);
    if (a.force_on && active) {
        const double2 ex = a.ftab[i], ey = a.ftab[a.g.nx + j];
        exy.x = ex.x * ey.x - ex.y * ey.y;
        exy.y = ex.x * ey.y + ex.y * ey.x;
    }
    const long long *const ring = m.sm + (threadIdx.y + R) * FXR + threadIdx.x + R;
    fx_u64 *const given = &m.sh->given[threadIdx.y >> 1], *const taken = &m.sh->taken[threadIdx.y >> 1];
    const int z0 = m.z0;
    for (int z = z0; z < m.z1; ++z) {
        if (!m.arrive()) break;
        const long long o =
            AC_BC(z * a.g.pxy + (long long)j * a.g.px + i, active ? a.g.elems : 1ll << 62, AC_BC_TILE_OUT);
        double f0[5] = {}, w0[5] = {};
        if (active) {
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                f0[q] = fx_load_now(a.fin[q] + o);
                if (!a.s0) w0[q] = fx_load_now(a.w[q] + o);
            }
        }
        long long GL[3], GU[3][3], u0[3];
        FxWide V[3] = {}, LU[3];
        long long GDs[3] = {0, 0, 0}, LUs[3];  // unequal spacing: over 2^8 and 2^6
        {
            const FxView Fl{ring, m.slot};
            const FxAxis l[3] = {fx_axis<0>(Fl), fx_axis<1>(Fl), fx_axis<2>(Fl)};
#pragma unroll
            for (int q = 0; q < 3; ++q) GL[q] = fx_first<ANISO>(l[q].d >> 2, fc, q);
        }
        {
            const FxView Fx{ring + FX_FIELD_TILE, m.slot}, Fy{ring + 2 * FX_FIELD_TILE, m.slot},
                Fz{ring + 3 * FX_FIELD_TILE, m.slot};
            u0[0] = Fx(0, 0, 0);
            u0[1] = Fy(0, 0, 0);
            u0[2] = Fz(0, 0, 0);
            if constexpr (ANISO) {
                fx_u_component_scaled<0>(Fx, u0[0], fc, GDs, GU[0], LUs[0]);
                fx_u_component_scaled<1>(Fy, u0[1], fc, GDs, GU[1], LUs[1]);
                fx_u_component_scaled<2>(Fz, u0[2], fc, GDs, GU[2], LUs[2]);
            } else {
                fx_u_component<0, EXT>(Fx, u0[0], V, GU[0], LU[0]);
                fx_u_component<1, EXT>(Fy, u0[1], V, GU[1], LU[1]);
                fx_u_component<2, EXT>(Fz, u0[2], V, GU[2], LU[2]);
            }
        }
        m.refill(z);
        FxSplit U[3], SL[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            U[q] = fx_split(u0[q] + Cu[q]);
            SL[q] = fx_split(GL[q]);
        }
        const long long div = GU[0][0] + GU[1][1] + GU[2][2];
        const double divu = fx_to_double(div, FX_EB64 + 2 + ku);
        const double adv_l = fx_to_double(fx_dot3(U, SL), FX_EB + 34 + ku + kl);
        fx_update(a, active, 0, o, f0[0], w0[0], -(fc.c1dt * adv_l) - fc.c1dt * divu);
        // viscosity, advection, 2 nu S . grad ln rho and the forcing
        double cph = 0.0;
        if (a.force_on) {
            const double2 ez = a.ftab[a.g.nx + a.g.ny + z];
            cph = exy.x * ez.x - exy.y * ez.y;
        }
        double ru[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const FxSplit g[3] = {fx_split(GU[q][0]), fx_split(GU[q][1]), fx_split(GU[q][2])};
            if (ANISO)
                ru[q] = fma(fc.nu180, fx_to_double(LUs[q], FX_EB64 + 6 + ku),
                            fc.nu2160 * fx_to_double(GDs[q], FX_EB64 + 8 + ku));
            else if (EXT)
                ru[q] = fma(fc.nu180, fx_to_double(fx_wide96(LU[q]), FX_EB + ku),
                            fc.nu2160 * fx_to_double(fx_wide96(V[q]), FX_EB + ku));
            else
                ru[q] = fc.nu2160 * fx_to_double(fx_wide96(V[q]), FX_EB + ku);
            ru[q] = fma(-fc.c1dt, fx_to_double(fx_dot3(U, g), FX_EB + 34 + 2 * ku), ru[q]);
            ru[q] = fma(fc.amp_dt[q], cph, ru[q]);
        }
        // the traceless rate of strain, X = 3/4 S
        double h;
        {
            FxSplit D[3], O[3];  // diagonal; xy, xz, yz
#pragma unroll
            for (int q = 0; q < 3; ++q) D[q] = fx_split((3 * GU[q][q] - div) >> 2);
            const long long xy = GU[0][1] + GU[1][0], xz = GU[0][2] + GU[2][0],
                            yz = GU[1][2] + GU[2][1];
            O[0] = fx_split((xy + (xy >> 1)) >> 2);
            O[1] = fx_split((xz + (xz >> 1)) >> 2);
            O[2] = fx_split((yz + (yz >> 1)) >> 2);
            const FxSplit r0[3] = {D[0], O[0], O[1]}, r1[3] = {O[0], D[1], O[2]},
                          r2[3] = {O[1], O[2], D[2]};
            const int eb = FX_EB + 36 + ku + kl;
            ru[0] = fma(fc.sg, fx_to_double(fx_dot3(r0, SL), eb), ru[0]);
            ru[1] = fma(fc.sg, fx_to_double(fx_dot3(r1, SL), eb), ru[1]);
            ru[2] = fma(fc.sg, fx_to_double(fx_dot3(r2, SL), eb), ru[2]);
            const Fx96 dd = fx_dot3(D, D), oo = fx_dot3(O, O);
            const fx_u64 low = (fx_u64)dd.low + 2ull * oo.low;
            Fx96 t;
            t.top = dd.top + 2 * oo.top + (long long)(low >> 32);
            t.low = (unsigned)low;
            h = fc.s2 * fx_to_double(t, FX_EB + 36 + 2 * ku);
        }
        if (EXT) h = fma(fc.inv_T_ref * fc.zeta_c1sq * divu, divu, h);
        // the other thread's terms
        m.ok = __all_sync(0xffffffffu, m.wait(given, (z - z0) & 1)) && m.ok;
        double x[FX_XCH];
#pragma unroll
        for (int q = 0; q < FX_XCH; ++q) x[q] = xch[q * FXT * FXT];
        __syncwarp();
        if ((threadIdx.x & 15) == 0 && (threadIdx.y & 1) == 0) fx_arrive(taken);
#pragma unroll
        for (int q = 0; q < 3; ++q)
            fx_update(a, active, 1 + q, o, f0[1 + q], w0[1 + q], ru[q] + x[q]);
        fx_update(a, active, 4, o, f0[4], w0[4], fma(x[5], h + x[3], x[4]));
        if (!m.ok) break;
        m.next();
    }
}

template <bool CFL, bool EXT, bool ANISO>
__global__ void __launch_bounds__(2 * FXT * FXT, 1)
    substep_fx_kernel(const SubstepArgs<double, double> a, const __grid_constant__ CUtensorMap map,
                      const FxCoefs fc, const FxPlan *plan, unsigned polls, int *err) {
    if (plan->kern != FX_GROUP) return;
    extern __shared__ __align__(128) unsigned char fx_smem[];
    __shared__ FxShared sh;
    fx_u64 *const etab = reinterpret_cast<fx_u64 *>(fx_smem + (size_t)FX_SLOTS * FX_PLANE_BYTES);
    double *const xch = reinterpret_cast<double *>(etab + 256) + threadIdx.y * FXT + threadIdx.x;
    const int tid = (threadIdx.z * FXT + threadIdx.y) * FXT + threadIdx.x;
    FxMarch m;
    m.map = &map;
    m.sm = reinterpret_cast<long long *>(fx_smem);
    m.sh = &sh;
    m.x0 = blockIdx.x * FXT;
    m.y0 = blockIdx.y * FXT;
    m.z0 = blockIdx.z * a.zchunk;
    m.z1 = min(m.z0 + a.zchunk, a.g.nz);
    if (tid == 0) {
        fx_u64 *const bars = sh.full;  // all of them, each for one arrival a phase
        for (int b = 0; b < FX_SLOTS + FX_WARPS; ++b)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(fx_smem_u32(bars + b))
                         : "memory");
        sh.done = 0;
        sh.fetched = FX_SLOTS;
        sh.polls = polls;
        if (CFL) {
            const double g = __longlong_as_double(
                (long long)*reinterpret_cast<volatile unsigned long long *>(a.cfl_max));
            sh.cfl_low = __float_as_int(g < 1e30 ? __double2float_rd(g) : 1e30f);
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        // padded plane z + d holds plane z - 3 + d: the planes z0 - 3 .. z0 + 3
        for (int d = 0; d < FX_SLOTS; ++d)
            fx_fetch(m.sm + d * FX_PLANE, &map, &sh.full[d], m.x0, m.y0, m.z0 + d);
    }
    for (int t = tid; t < 256; t += 2 * FXT * FXT) etab[t] = EXP_FIX[t];
    __syncthreads();
#pragma unroll
    for (int d = 0; d < FX_SLOTS; ++d) m.slot[d] = d * FX_PLANE;
    m.ok = true;
    for (int d = 0; d < FX_SLOTS - 1; ++d) m.ok = fx_wait(&sh.full[d], 0, polls) && m.ok;
    m.ok = __all_sync(0xffffffffu, m.ok);
    m.last = FX_SLOTS - 1;
    m.parity = 0;
    double cfl = 0.0;
    const int i = m.x0 + threadIdx.x, j = m.y0 + threadIdx.y;
    if (m.ok) {
        if (threadIdx.z)
            fx_march_a<CFL, EXT, ANISO>(a, fc, plan, etab, xch, m, i, j, cfl);
        else
            fx_march_u<EXT, ANISO>(a, fc, plan, xch, m, i, j);
    }
    // a wait that ran out is reported, and no copy may be in flight when the CTA ends: with
    // every warp out of the march no plane is asked for any more, and the last fill of
    // each slot is waited for
    if (__syncthreads_or(!m.ok) && tid == 0) {
        *reinterpret_cast<volatile int *>(err) = 1;  // page-locked host memory
        for (unsigned n = sh.fetched - FX_SLOTS; n < sh.fetched; ++n)
            fx_wait(&sh.full[n % FX_SLOTS], (n / FX_SLOTS) & 1, FX_WAIT_LIMIT);
    }
    if (CFL) block_max_to_global(cfl, a.cfl_max);
}

// What substep_fx_kernel does not take: FX_FIELD (FORM FX_EQUAL) and FX_PLAIN, plain
// binary64 stencils, the arithmetic of AC_STENCIL_FP64.  Launched every substep beside
// substep_fx_kernel (its own register allocation: with the group body in one kernel
// ptxas spilled); whichever the plan did not choose returns at once, which costs a
// small grid 3.7 us a launch, so these two share one.  Two CTAs of 128 threads per SM
// (8 warps, as many as 255 registers allow).
template <bool CFL, bool EXT, int FORM>
__global__ void __launch_bounds__(128, 2) substep_fx_fallback_kernel(const SubstepArgs<double, double> a,
                                                                     const FxPtrs fx, FxCoefs fc,
                                                                     const FxPlan *plan) {
    using IX = typename FxIndex<FORM>::type;
    const int kern = plan->kern;
    if (kern == FX_GROUP) return;
    if (FORM == FX_UNEQUAL || kern == FX_PLAIN) {
        substep_body<double, double, IdxPeriodic32, CFL, 3, EXT>(a);
        return;
    }
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const bool active = i < a.g.nx && j < a.g.ny;
    __shared__ double etab[512];
    exp_tab_stage(etab);
    double cfl = 0.0;
    if (active) fx_column<true, IX, CFL, EXT>(a, fx, fc, plan, etab, i, j, cfl);
    if (CFL) block_max_to_global(cfl, a.cfl_max);
}

// The columns' FX_GROUP, for boxes too thin for the 16 x 16 tiles (fx_form).
template <bool CFL, bool EXT>
__global__ void __launch_bounds__(128, 2) substep_fx_column_kernel(const SubstepArgs<double, double> a,
                                                                   const FxPtrs fx, FxCoefs fc,
                                                                   const FxPlan *plan) {
    if (plan->kern != FX_GROUP) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const bool active = i < a.g.nx && j < a.g.ny;
    __shared__ double etab[512];
    exp_tab_stage(etab);
    double cfl = 0.0;
    if (active) fx_column<false, IdxPeriodic32, CFL, EXT>(a, fx, fc, plan, etab, i, j, cfl);
    if (CFL) block_max_to_global(cfl, a.cfl_max);
}

}  // namespace ac
