// FP64 substep: exact integer stencil sums on cubic periodic grids (the fast
// path), plain binary64 stencil arithmetic otherwise.
#include <cmath>
#include <type_traits>

#include <cudaTypedefs.h>

#include "substep_fx.cuh"

namespace ac {

static unsigned fx_grid(long long n) {  // n work items of one thread each
    long long b = (n + 255) / 256;
    return (unsigned)(b > 152 * 8 ? 152 * 8 : (b < 1 ? 1 : b));
}

// z extent of a CTA's march in the tiled kernel (one CTA per SM): the one with the
// fewest plane steps over all waves, a CTA's start counted as one more step.
static int fx_zchunk(long long tiles, int nz) {
    int best = nz;
    long long cost = -1;
    for (int c = 1; c <= nz && c <= 1024; ++c) {
        const int zc = (nz + c - 1) / c;
        const long long ctas = tiles * ((nz + zc - 1) / zc);
        const long long t = ((ctas + 151) / 152) * (zc + 1);
        if (cost < 0 || t < cost) {
            cost = t;
            best = zc;
        }
        if (tiles * c > 152ll * 64) break;
    }
    return best;
}

// Launch shape of the kernels that go column by column: threads of (32, 4) cells, enough
// z-slices for several waves of CTAs, up to 16 cells per thread.
static int fx_column_zchunk(const Geom &g) {
    const long long xy = (long long)((g.nx + 31) / 32) * ((g.ny + 3) / 4);
    const long long z = xy * g.nz / (8 * 152);
    return (int)(z < 1 ? 1 : (z > 16 ? 16 : z));
}

// Which form the box's shape asks for.  Tiles of 16 x 16 cells and copies padded by three
// cells on each side suit boxes with extent in every direction; a thin box pads them away.
// The times of either, in us, from what one plane takes (GB300, 54 boxes from one cell to
// 2048^2 x 8, equal spacing and ratios of 1.25, within a fifth or so): a CTA of the tiles
// takes 8.6 a plane (unequal 10.8) and one more to start; a pair of column CTAs on an SM
// 8.5 to 16.4 a plane by its rows and 4.6 to start (plain stencils 16.5 to 41 and 7.5);
// the copies 23 us a million cells, the columns' 17.
int fx_form(const Geom &g, bool equal) {
    const long long tiles = (long long)((g.nx + FXT - 1) / FXT) * ((g.ny + FXT - 1) / FXT);
    const int zc = fx_zchunk(tiles, g.nz), rows = g.ny < 4 ? g.ny : 4;
    const double waves = (double)((tiles * ((g.nz + zc - 1) / zc) + 151) / 152);
    const double mcells = 1e-6 * g.elems;
    const double mpadded = 1e-6 * (g.nx + 2 * R) * (double)(g.ny + 2 * R) * (g.nz + 2 * R);
    const double tile = 4.0 + 23.0 * mpadded + waves * (zc + 1) * (equal ? 8.6 : 10.8);
    static const double group[4] = {8.5, 13.2, 15.0, 16.4}, plain[4] = {16.5, 22.0, 32.0, 41.0};
    const int cz = fx_column_zchunk(g);
    const long long blocks = (long long)((g.nx + 31) / 32) * ((g.ny + 3) / 4) * ((g.nz + cz - 1) / cz);
    const double pairs = blocks < 304 ? 1.0 : blocks / 304.0;
    if (equal)
        return tile <= 6.0 + 17.0 * mcells + pairs * (4.6 + cz * group[rows - 1]) ? FX_EQUAL : FX_COLUMNS;
    // Unequal spacing: below 16384 cells, or with no more than one CTA of plain stencils to an
    // SM, preparation is what counts (24^3 93 us a step plain, some 118 with tiles, 60x20x14
    // 94 against 125); from there on the model decides, small boxes with a full row of a tile
    // aside (26^3 118 against 158, 17x31x33 119 against 158, but 16x1x1100 332 against 293).
    if (g.elems < 16384 || blocks <= 152) return FX_NONE;
    return (g.elems < 32768 && g.nx >= FXT) || 17.0 + tile <= pairs * (7.5 + cz * plain[rows - 1])
               ? FX_UNEQUAL
               : FX_NONE;
}

// Padded row length (even: the strides of the tensor map are multiples of 16 bytes), the
// geometry of the int64 copies, their bytes, and the tensor map over the padded ones: dims
// (px, py, pz, field), box one plane of a tile with its halo, all fields.
static int fx_px(const Geom &g) { return (g.nx + 2 * R + 1) & ~1; }
static Geom fx_geom(const Geom &g, int form) {
    Geom c = g;
    if (form == FX_COLUMNS) return c;
    c.px = fx_px(g);
    c.pxy = (long long)c.px * (g.ny + 2 * R);
    c.origin = R * c.pxy + (long long)R * c.px + R;
    c.elems = c.pxy * (g.nz + 2 * R);
    return c;
}
size_t fx_copy_bytes(const Geom &g, int form) {
    return (size_t)NF * fx_geom(g, form).elems * sizeof(long long);
}
cudaError_t fx_encode_map(void *base, const Geom &g, CUtensorMap *map) {
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    cudaError_t e =
        cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess) return e;
    if (q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
    auto enc = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    const cuuint64_t px = fx_px(g), py = g.ny + 2 * R, pz = g.nz + 2 * R;
    const cuuint64_t dims[4] = {px, py, pz, NF};
    const cuuint64_t strides[3] = {8 * px, 8 * px * py, 8 * px * py * pz};
    const cuuint32_t box[4] = {FXR, FXR, 1, NF};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 4, base, dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <bool CFL, bool EXT, bool ANISO>
static cudaError_t launch_fx_group(SubstepArgs<double, double> a, const CUtensorMap &map,
                                   const FxCoefs &fc, const FxPlan *plan, unsigned polls, int *err,
                                   cudaStream_t st) {
    auto k = substep_fx_kernel<CFL, EXT, ANISO>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FX_SMEM);
    if (e != cudaSuccess) return e;
    const unsigned gx = (a.g.nx + FXT - 1) / FXT, gy = (a.g.ny + FXT - 1) / FXT;
    a.zchunk = fx_zchunk((long long)gx * gy, a.g.nz);
    const dim3 grid(gx, gy, (a.g.nz + a.zchunk - 1) / a.zchunk);
    k<<<grid, dim3(FXT, FXT, 2), FX_SMEM, st>>>(a, map, fc, plan, polls, err);
    return cudaGetLastError();
}

cudaError_t launch_substep_f64(const SubstepLaunch &L, cudaStream_t st, int *launches) {
    // Integer sums need 32-bit neighbour offsets (always true for a binary64
    // state in HBM: fewer than 2^31 cells per array); their kernels fold dt into
    // the coefficients, so a step of zero or of extreme magnitude (1 / dt^2 out of
    // range) takes the plain binary64 stencils.
    const double adt = fabs(L.dt);
    if (!L.use_fx || L.g.elems >= (1ll << 31) || !(adt >= 1e-100 && adt <= 1e100))
        return launch_substep_t<double, double>(L, st, launches);
    SubstepArgs<double, double> a;
    a.g = L.g;
    FxPtrs fx;
    for (int q = 0; q < NF; ++q) {
        a.fin[q] = static_cast<const double *>(L.fin[q]);
        a.fout[q] = static_cast<double *>(L.fout[q]);
        a.w[q] = static_cast<double *>(L.w[q]);
        fx.f[q] = a.fin[q];
    }
    fx.halo = L.use_fx == FX_COLUMNS ? 0 : R;
    fx.py = L.g.ny + 2 * fx.halo;
    fx.g = fx_geom(L.g, L.use_fx);
    for (int q = 0; q < NF; ++q) fx.F[q] = static_cast<long long *>(L.fx_copies) + q * fx.g.elems;
    a.k = to_dev<double>(L.c, L.ph);
    a.alpha = L.alpha;
    a.beta = L.beta;
    a.dt = L.dt;
    a.s0 = L.s == 0;
    a.force_on = L.force.on;
    a.ftab = L.force.tab;
    for (int m = 0; m < 3; ++m) a.amp_e[m] = L.force.amp_e[m];
    a.cfl_max = L.cfl_max;
    // the step folded into the RHS coefficients; with unequal spacing they hold the
    // smallest one and the numerators carry the ratios
    const bool aniso = L.use_fx == FX_UNEQUAL;
    const double h = fmin(L.dx[0], fmin(L.dx[1], L.dx[2]));
    FxCoefs fc = {};
    if (aniso) {
        const int pa[3] = {0, 0, 1}, pb[3] = {1, 2, 2};
        for (int m = 0; m < 3; ++m) {
            const double r = h / L.dx[m];
            fx_fraction(r, &fc.r1h[m], &fc.r1l[m]);
            fx_fraction(r * r, &fc.r2h[m], &fc.r2l[m]);
            fx_fraction((h / L.dx[pa[m]]) * (h / L.dx[pb[m]]), &fc.rmh[m], &fc.rml[m]);
        }
    }
    const double dts = L.dt;
    const double c1 = 1.0 / (60.0 * h);
    fc.c1dt = dts * c1;
    fc.nu180 = dts * (L.ph.nu / (180.0 * h * h));
    fc.nu2160 = dts * ((L.ph.nu + 3.0 * L.ph.zeta) / (2160.0 * h * h));
    fc.inv180dx2 = 1.0 / (180.0 * h * h);
    fc.inv720dx2 = 1.0 / (720.0 * h * h);
    fc.two_nu_c1sq = dts * (2.0 * L.ph.nu * c1 * c1);
    fc.K_c1sq = dts * (L.ph.K * c1 * c1);
    fc.zeta_c1sq = dts * (L.ph.zeta * c1 * c1);
    fc.eta_dt = dts * a.k.eta;
    fc.hc_dt = dts * a.k.hc;
    fc.K_dt = dts * a.k.K;
    for (int m = 0; m < 3; ++m) fc.amp_dt[m] = dts * L.force.amp_e[m];
    fc.inv_dt2 = 1.0 / (dts * dts);
    fc.sg = fc.two_nu_c1sq * (4.0 / 3.0);
    fc.inv_T_ref = a.k.inv_T_ref;
    fc.s2 = fc.two_nu_c1sq * (16.0 / 9.0) * fc.inv_T_ref;
    fc.jb = -fc.c1dt * fc.inv720dx2;
    fc.j2 = fc.eta_dt * fc.inv720dx2 * fc.inv720dx2 * fc.inv_T_ref;
    fc.eta180 = fc.eta_dt * fc.inv180dx2;
    fc.c1sq = c1 * c1;
    fc.c1f = nextafterf((float)c1, INFINITY);
    fc.cs2_ref_f = nextafterf((float)a.k.cs2_ref, INFINITY);

    const long long n = L.g.elems;
    FxPlan *plan = static_cast<FxPlan *>(L.fx_plan);
    cudaError_t e;
    fx_stats_kernel<<<fx_grid(n / 2), 256, 0, st>>>(fx, n, L.fx_stats, plan, L.ph.gamma_cp, L.ph.gm1,
                                                   L.use_fx);
    if (fx.g.elems > 256ll * 152 * 8)
        fx_quantize_kernel<2><<<fx_grid((fx.g.elems + 1) / 2), 256, 0, st>>>(fx, L.g, plan);
    else
        fx_quantize_kernel<1><<<fx_grid(fx.g.elems), 256, 0, st>>>(fx, L.g, plan);
    if (L.ev_mid) {
        e = cudaEventRecord(L.ev_mid, st);
        if (e != cudaSuccess) return e;
    }

    const dim3 block(32, 4, 1);
    a.zchunk = fx_column_zchunk(L.g);
    const dim3 grid((L.g.nx + 31) / 32, (L.g.ny + 3) / 4, (L.g.nz + a.zchunk - 1) / a.zchunk);
    const bool ext = L.ph.ext(), cfl = a.cfl_max != nullptr;
    // one kernel per plan; those the plan did not choose return at once
    auto launch = [&](auto c, auto x) -> cudaError_t {
        constexpr bool C = decltype(c)::value, X = decltype(x)::value;
        if (L.use_fx == FX_COLUMNS) {
            substep_fx_column_kernel<C, X><<<grid, block, 0, st>>>(a, fx, fc, plan);
            substep_fx_fallback_kernel<C, X, FX_COLUMNS><<<grid, block, 0, st>>>(a, fx, fc, plan);
            return cudaSuccess;
        }
        const cudaError_t r =
            aniso ? launch_fx_group<C, X, true>(a, *L.fx_map, fc, plan, L.fx_polls, L.fx_err, st)
                  : launch_fx_group<C, X, false>(a, *L.fx_map, fc, plan, L.fx_polls, L.fx_err, st);
        if (r != cudaSuccess) return r;
        if (aniso) substep_fx_fallback_kernel<C, X, FX_UNEQUAL><<<grid, block, 0, st>>>(a, fx, fc, plan);
        else substep_fx_fallback_kernel<C, X, FX_EQUAL><<<grid, block, 0, st>>>(a, fx, fc, plan);
        return cudaSuccess;
    };
    using yes = std::true_type;
    using no = std::false_type;
    e = ext ? (cfl ? launch(yes(), yes()) : launch(no(), yes()))
            : (cfl ? launch(yes(), no()) : launch(no(), no()));
    if (e != cudaSuccess) return e;
    *launches += 4;
    return cudaGetLastError();
}

// Size of the device plan of the integer-sum path (allocated by the handle).
size_t fx_plan_bytes() { return sizeof(FxPlan); }

// Substeps counted in each mode, or (ran) that each form ran, read from a plan.
cudaError_t fx_plan_counts(const void *plan, bool ran, unsigned long long *counts, cudaStream_t st) {
    const FxPlan *p = static_cast<const FxPlan *>(plan);
    cudaError_t e = cudaMemcpyAsync(counts, ran ? p->ran : p->taken,
                                    (ran ? 4 : 3) * sizeof(unsigned long long),
                                    cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return e;
}

// The table-driven exp of the binary64 kernels beside CUDA's exp, for tests:
// y[i] = exp_tab(x[i]), y[n + i] = exp(x[i]), y[2n + i] and y[3n + i] = the pair
// exp(x[i]), exp(-x[i]) from exp_tab_pm; where exp_tab_ok(x[i]) fails, the three
// table values are CUDA's (the kernels' fallback).
__global__ void diag_exp_kernel(const double *x, long long n, double *y) {
    __shared__ double tab[512];
    exp_tab_stage(tab);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const double v = x[i];
        double a, b, c;
        if (exp_tab_ok(v)) {
            a = exp_tab(v, tab);
            exp_tab_pm(v, tab, b, c);
        } else {
            a = exp(v);
            b = exp(v);
            c = exp(-v);
        }
        y[i] = a;
        y[n + i] = exp(v);
        y[2 * n + i] = b;
        y[3 * n + i] = c;
    }
}

}  // namespace ac

extern "C" int ac_diag_exp_table(const double *x, long long n, double *y, void *stream) {
    if (n < 0 || (n > 0 && (!x || !y))) return AC_ERR_ARG;
    if (n == 0) return AC_OK;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const long long want = (n + 255) / 256;
    const unsigned blocks = (unsigned)(want < 152 * 8 ? want : 152 * 8);
    ac::diag_exp_kernel<<<blocks, 256, 0, st>>>(x, n, y);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return e == cudaSuccess ? AC_OK : ac::ac_report_cuda(e);
}

AC_BC_READER(bc_take_f64)
