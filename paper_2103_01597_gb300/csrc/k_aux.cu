// Auxiliary kernels: periodic halo fill (Sec. 3.3), forcing phase tables,
// host-format staging (load/store with precision conversion), and binary64
// reductions of fields and derived quantities.
#include <float.h>
#include <math.h>

#include "fx_arith.cuh"
#include "reduce.cuh"

namespace ac {

// ---------------------------------------------------------------------------
// Coefficients (host).  Central weights of order 2r on the points of Eq. 13
// (axes and face diagonals out to radius r), as integer numerators over a
// common denominator:
//   r = 3 (Sec. 4): d/dx (45, -9, 1) / 60 on (f_m - f_-m); d2/dx2 -49/18 on f_0
//          and (3/2, -3/20, 1/90) on (f_m + f_-m); d2/dxdy (270, -27, 2) / 720
//          on the diagonal sums S_m;
//   r = 1: (1) / 2;   -2, (1);                       (1) / 4;
//   r = 2: (8, -1) / 12;   -30/12, (16, -1) / 12;    (16, -1) / 48;
//   r = 4: (672, -168, 32, -3) / 840;   -14350/5040, (8064, -1008, 128, -9) / 5040;
//          (8064, -1008, 128, -9) / 20160.
// The mixed weights are the second-difference weights over 4 (S_m expands like
// 4 m^2 dx_a dx_b d_a d_b plus the same higher moments).
// ---------------------------------------------------------------------------
StencilCoefs make_coefs(const double dx[3], int radius) {
    StencilCoefs c = {};
    c.radius = radius;
    const int pa[3] = {0, 0, 1}, pb[3] = {1, 2, 2};
    if (radius == 3) {
        const double w1[3] = {45.0, -9.0, 1.0};
        const double w2[3] = {1.5, -0.15, 1.0 / 90.0};
        const double wc[3] = {270.0, -27.0, 2.0};
        for (int a = 0; a < 3; ++a) {
            for (int m = 0; m < 3; ++m) c.d1[a][m] = w1[m] / (60.0 * dx[a]);
            c.d2[a][0] = (-49.0 / 18.0) / (dx[a] * dx[a]);
            for (int m = 0; m < 3; ++m) c.d2[a][m + 1] = w2[m] / (dx[a] * dx[a]);
        }
        for (int pl = 0; pl < 3; ++pl)
            for (int m = 0; m < 3; ++m) c.dc[pl][m] = wc[m] / (720.0 * dx[pa[pl]] * dx[pb[pl]]);
        return c;
    }
    static const double n1[5][4] = {{0}, {1}, {8, -1}, {0}, {672, -168, 32, -3}};
    static const double q1[5] = {0, 2, 12, 0, 840};
    static const double n2[5][5] = {{0}, {-2, 1}, {-30, 16, -1}, {0}, {-14350, 8064, -1008, 128, -9}};
    static const double q2[5] = {0, 1, 12, 0, 5040};
    for (int a = 0; a < 3; ++a) {
        for (int m = 0; m < radius; ++m) c.d1[a][m] = n1[radius][m] / (q1[radius] * dx[a]);
        for (int m = 0; m <= radius; ++m) c.d2[a][m] = n2[radius][m] / (q2[radius] * dx[a] * dx[a]);
    }
    for (int pl = 0; pl < 3; ++pl)
        for (int m = 0; m < radius; ++m)
            c.dc[pl][m] = n2[radius][m + 1] / (4.0 * q2[radius] * dx[pa[pl]] * dx[pb[pl]]);
    return c;
}

PhysConsts make_phys(const ac_params &p) {
    PhysConsts c;
    c.nu = p.nu;
    c.eta = p.eta;
    c.inv_cp = 1.0 / p.cp;
    c.cs2_ref = p.cs0 * p.cs0 * exp(-(p.gamma - 1.0) * p.lnrho0);
    c.gamma_cp = p.gamma / p.cp;
    c.gm1 = p.gamma - 1.0;
    c.cp_gm1 = p.cp * (p.gamma - 1.0);
    c.K = 0.0;
    c.zeta = 0.0;
    c.hc = 0.0;
    return c;
}

// ---------------------------------------------------------------------------
// Periodic halo of the padded layout: every halo cell takes the value of its
// image ((s - r) mod n) + r per axis.  Halo cells are enumerated as three
// disjoint groups: the z-slabs (full padded planes), the y-slabs of the
// interior z range, and the x-slabs of the interior y and z ranges.
// ---------------------------------------------------------------------------

template <typename T>
__global__ void halo_kernel_pack(PtrPack<T> pk, Geom g, long long nz_slab, long long ny_slab,
                                 long long total) {
    T *arr = pk.p[blockIdx.y];
    const int mx = g.px;
    const int my = (int)(g.pxy / g.px);
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        int i, j, k;
        if (t < nz_slab) {
            const long long plane = (long long)mx * my;
            const long long zs = t / plane;
            const long long rem = t - zs * plane;
            k = zs < R ? (int)zs : (int)(g.nz + zs);
            j = (int)(rem / mx);
            i = (int)(rem - (long long)j * mx);
        } else if (t < nz_slab + ny_slab) {
            const long long u = t - nz_slab;
            const long long row = (long long)mx * 2 * R;
            const long long kz = u / row;
            const long long rem = u - kz * row;
            const int ys = (int)(rem / mx);
            k = (int)kz + R;
            j = ys < R ? ys : g.ny + ys;
            i = (int)(rem - (long long)ys * mx);
        } else {
            const long long u = t - nz_slab - ny_slab;
            const long long kz = u / ((long long)g.ny * 2 * R);
            const long long rem = u - kz * ((long long)g.ny * 2 * R);
            const int jy = (int)(rem / (2 * R));
            const int xs = (int)(rem - (long long)jy * 2 * R);
            k = (int)kz + R;
            j = jy + R;
            i = xs < R ? xs : g.nx + xs;
        }
        const int si = wrap_near(i - R, g.nx) + R;
        const int sj = wrap_near(j - R, g.ny) + R;
        const int sk = wrap_near(k - R, g.nz) + R;
        arr[(long long)k * g.pxy + (long long)j * mx + i] =
            arr[(long long)sk * g.pxy + (long long)sj * mx + si];
    }
}

cudaError_t launch_halo(int precision, const Geom &g, void *const f[NF], cudaStream_t st) {
    if (!g.padded) return cudaSuccess;
    const long long mx = g.px, my = g.pxy / g.px;
    const long long nz_slab = 2LL * R * mx * my;
    const long long ny_slab = (long long)g.nz * 2 * R * mx;
    const long long nx_slab = (long long)g.nz * g.ny * 2 * R;
    const long long total = nz_slab + ny_slab + nx_slab;
    long long blocks = (total + 255) / 256;
    if (blocks > 152 * 8) blocks = 152 * 8;
    const dim3 grid((unsigned)blocks, NF);
    if (precision == AC_FP64) {
        PtrPack<double> pk;
        for (int q = 0; q < NF; ++q) pk.p[q] = static_cast<double *>(f[q]);
        halo_kernel_pack<double><<<grid, 256, 0, st>>>(pk, g, nz_slab, ny_slab, total);
    } else {
        PtrPack<float> pk;
        for (int q = 0; q < NF; ++q) pk.p[q] = static_cast<float *>(f[q]);
        halo_kernel_pack<float><<<grid, 256, 0, st>>>(pk, g, nz_slab, ny_slab, total);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Forcing tables: e^{i 2 pi k_a i / n_a} per axis (binary64, then a binary32
// copy), with the phase phi folded into the z table.  Layout: [nx | ny | nz]
// double2 entries, followed by the same count of float2 entries.
// ---------------------------------------------------------------------------
__global__ void forcing_table_kernel(int nx, int ny, int nz, int kx, int ky, int kz,
                                     double cphi, double sphi, double2 *tab) {
    const int total = nx + ny + nz;
    float2 *tabf = reinterpret_cast<float2 *>(tab + total);
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        int n, kk, i;
        if (t < nx) {
            n = nx; kk = kx; i = t;
        } else if (t < nx + ny) {
            n = ny; kk = ky; i = t - nx;
        } else {
            n = nz; kk = kz; i = t - nx - ny;
        }
        long long m = ((long long)kk * i) % n;
        if (m < 0) m += n;
        double s, c;
        sincospi(2.0 * (double)m / (double)n, &s, &c);
        if (t >= nx + ny) {  // rotate by phi
            const double c2 = c * cphi - s * sphi;
            const double s2 = s * cphi + c * sphi;
            c = c2;
            s = s2;
        }
        tab[t] = make_double2(c, s);
        tabf[t] = make_float2((float)c, (float)s);
    }
}

cudaError_t launch_forcing_table(const Geom &g, const int k[3], double phi, double2 *tab,
                                 cudaStream_t st) {
    const int total = g.nx + g.ny + g.nz;
    const int blocks = (total + 255) / 256;
    forcing_table_kernel<<<blocks, 256, 0, st>>>(g.nx, g.ny, g.nz, k[0], k[1], k[2], cos(phi),
                                                 sin(phi), tab);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Staging: an unpadded float64 slab of nzc z-planes starting at z0 <-> a
// device array in its layout and precision.
// ---------------------------------------------------------------------------
// Host-format staging (S: binary64 or binary32, unpadded planes z0 .. z0 + nzc)
// to and from a device array of element type T in the handle's layout.
template <typename S, typename T>
__global__ void scatter_kernel(const S *__restrict__ stage, T *__restrict__ dst, Geom g, int z0,
                               long long count) {
    const long long plane = (long long)g.nx * g.ny;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < count;
         t += (long long)gridDim.x * blockDim.x) {
        const long long kz = t / plane;
        const long long rem = t - kz * plane;
        const long long j = rem / g.nx;
        const long long i = rem - j * g.nx;
        dst[g.origin + (z0 + kz) * g.pxy + j * g.px + i] = (T)stage[t];
    }
}

template <typename T, typename S>
__global__ void gather_kernel(const T *__restrict__ src, Geom g, int z0, long long count,
                              S *__restrict__ stage) {
    const long long plane = (long long)g.nx * g.ny;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < count;
         t += (long long)gridDim.x * blockDim.x) {
        const long long kz = t / plane;
        const long long rem = t - kz * plane;
        const long long j = rem / g.nx;
        const long long i = rem - j * g.nx;
        stage[t] = (S)src[g.origin + (z0 + kz) * g.pxy + j * g.px + i];
    }
}

static unsigned grid_for(long long count) {
    long long b = (count + 255) / 256;
    return (unsigned)(b > 152 * 16 ? 152 * 16 : (b < 1 ? 1 : b));
}

template <typename S>
static cudaError_t scatter_t(const S *stage, void *dst, int elem_size, const Geom &g, int z0,
                             int nzc, cudaStream_t st) {
    const long long count = (long long)g.nx * g.ny * nzc;
    if (elem_size == 8)
        scatter_kernel<S, double><<<grid_for(count), 256, 0, st>>>(stage, (double *)dst, g, z0, count);
    else
        scatter_kernel<S, float><<<grid_for(count), 256, 0, st>>>(stage, (float *)dst, g, z0, count);
    return cudaGetLastError();
}

template <typename S>
static cudaError_t gather_t(const void *src, int elem_size, const Geom &g, int z0, int nzc,
                            S *stage, cudaStream_t st) {
    const long long count = (long long)g.nx * g.ny * nzc;
    if (elem_size == 8)
        gather_kernel<double, S><<<grid_for(count), 256, 0, st>>>((const double *)src, g, z0, count,
                                                                 stage);
    else
        gather_kernel<float, S><<<grid_for(count), 256, 0, st>>>((const float *)src, g, z0, count,
                                                                stage);
    return cudaGetLastError();
}

cudaError_t launch_scatter(const double *stage, void *dst, int elem_size, const Geom &g, int z0,
                           int nzc, cudaStream_t st) {
    return scatter_t(stage, dst, elem_size, g, z0, nzc, st);
}
cudaError_t launch_gather(const void *src, int elem_size, const Geom &g, int z0, int nzc,
                          double *stage, cudaStream_t st) {
    return gather_t(src, elem_size, g, z0, nzc, stage, st);
}
cudaError_t launch_scatter_f32(const float *stage, void *dst, int elem_size, const Geom &g, int z0,
                               int nzc, cudaStream_t st) {
    return scatter_t(stage, dst, elem_size, g, z0, nzc, st);
}
cudaError_t launch_gather_f32(const void *src, int elem_size, const Geom &g, int z0, int nzc,
                              float *stage, cudaStream_t st) {
    return gather_t(src, elem_size, g, z0, nzc, stage, st);
}

// ---------------------------------------------------------------------------
// Reductions in binary64.  Each block reduces its share of the cells into
// partials[block] and flags[block] (non-finite seen); the last block to finish combines
// the partials in a fixed order, so results are deterministic for a given grid, and
// writes them to the device and to page-locked host memory.
//
// Three kernels.  Quantities of the cell alone (fields, |u|, E_K) stream through
// reduce_cells_kernel, bound by memory.  E_M sums and, in binary32, the CFL speed go
// through reduce_curl_kernel, whose threads march along z (the periodic offsets of x and
// y are set once).  In binary64 an FP64-pipe instruction costs a warp about 78 cycles, so
// the six derivatives of the curl are taken in integers there (fx_arith.cuh).  The
// largest CFL speed (reduce_cfl_max_kernel) is searched with a binary32 upper bound, exact
// binary64 speeds only where it exceeds the largest known.
// The rest (max and min of E_K and E_M, other orders, CFL sums) takes the general kernel.
// Measured at 256^3 in binary64, host time of one call each: E_K 245 us, E_M 930 (883 with
// one scale for all 36 values, which lost bits to uniform parts of A), rms |u| 145, the
// CFL speed 1196, min ln rho 58, together 2580 (6470 all through the general kernel).
// ---------------------------------------------------------------------------
constexpr int RED_THREADS = 256;
constexpr int RED_MAX_BLOCKS = 8 * 152;  // eight 256-thread CTAs per SM

int reduce_max_blocks() { return RED_MAX_BLOCKS; }

struct RedOut {
    double *partials;
    unsigned int *flags;    // [RED_MAX_BLOCKS] and the count of finished blocks
    double *dev, *host;     // value and flag word
};

__device__ __forceinline__ void red_write(const RedOut &o, double r, unsigned int bad) {
    o.dev[0] = r;
    reinterpret_cast<unsigned int *>(o.dev + 1)[0] = bad;
    *reinterpret_cast<volatile double *>(o.host) = r;
    *reinterpret_cast<volatile unsigned int *>(o.host + 1) = bad;
}

// Whether this block is the last of the grid to get here (every thread's earlier writes
// are then visible to the last block); the counter is left at zero.
__device__ __forceinline__ bool red_last_block(unsigned int *counter) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x + threadIdx.y == 0)
        last = atomicInc(counter, gridDim.x - 1) == gridDim.x - 1;
    __syncthreads();
    return last;
}

// Combine a block's values; then, in the grid's last block, the partials.  ROOT: the
// result is the square root, in R, of the combined value (max or min of |u| from |u|^2).
template <typename R>
__device__ void red_finish(const RedOut &o, int op, double acc, unsigned int bad, double count,
                           bool root) {
    __shared__ double sh[RED_THREADS / 32];
    __shared__ unsigned int shb[RED_THREADS / 32];
    const int tid = threadIdx.y * blockDim.x + threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int pass = 0; pass < 2; ++pass) {
#pragma unroll
        for (int k = 16; k > 0; k >>= 1) {
            acc = red_combine(op, acc, __shfl_down_sync(0xffffffffu, acc, k));
            bad |= __shfl_down_sync(0xffffffffu, bad, k);
        }
        if (lane == 0) {
            sh[wid] = acc;
            shb[wid] = bad;
        }
        __syncthreads();
        double r = sh[0];
        unsigned int b = shb[0];
        if (tid == 0)
            for (int w = 1; w < RED_THREADS / 32; ++w) {
                r = red_combine(op, r, sh[w]);
                b |= shb[w];
            }
        if (pass == 1) {
            if (tid == 0) {
                if (op == AC_RMS) r = sqrt(r / count);
                if (root && r >= 0.0) r = (double)(R)sqrt((R)r);
                red_write(o, r, b);
            }
            return;
        }
        if (tid == 0) {
            o.partials[blockIdx.x] = r;
            o.flags[blockIdx.x] = b;
        }
        if (!red_last_block(o.flags + RED_MAX_BLOCKS)) return;
        acc = red_init(op);
        bad = 0;
        for (int t = tid; t < (int)gridDim.x; t += RED_THREADS) {
            acc = red_combine(op, acc, __ldcg(o.partials + t));
            bad |= __ldcg(o.flags + t);
        }
    }
}

// Rows of constant (y, z) are dealt to warps; lanes walk x.  The periodic
// offsets of y and z are set once per row, those of x once per cell.
template <typename R, class IX, int RAD = 3>
__global__ void __launch_bounds__(RED_THREADS) reduce_kernel(PtrPack<const R> pk, Geom g,
                                                             DevCoefs<R> k, int op, int quantity,
                                                             double count, RedOut out) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const long long rows = (long long)g.ny * g.nz;
    double acc = red_init(op);
    unsigned int bad = 0;
    for (long long row = (long long)blockIdx.x * (RED_THREADS / 32) + wid; row < rows;
         row += (long long)gridDim.x * (RED_THREADS / 32)) {
        const int kz = (int)(row / g.ny);
        const int j = (int)(row - (long long)kz * g.ny);
        IX ix;
        ix.set_xy(0, j, g);
        ix.set_z(kz, g);
        for (int i = lane; i < g.nx; i += 32) {
            ix.set_x(i, g);
            const double v = cell_quantity<R, IX, RAD>(pk.p, ix, k, quantity);
            if (!isfinite(v)) bad = 1;
            acc = red_combine(op, acc, op == AC_RMS ? v * v : v);
        }
    }
    red_finish<R>(out, op, acc, bad, count, false);
}

// Largest or smallest value met, NaN left out (as fmax and fmin leave it): binary32 by the
// FP32 pipe, binary64 by integer keys ordered like the values.
struct RedExtreme32 {
    float v;
    int max;
    __device__ RedExtreme32(int op) : v(op == AC_MAX ? -INFINITY : INFINITY), max(op == AC_MAX) {}
    __device__ void add(float x) { v = max ? fmaxf(v, x) : fminf(v, x); }
    __device__ double get() const { return (double)v; }
};
struct RedExtreme64 {
    long long key;
    int max;
    __device__ static long long order(long long b) { return b ^ ((b >> 63) & 0x7fffffffffffffffll); }
    __device__ RedExtreme64(int op) : max(op == AC_MAX) {  // an infinity: combines with any value
        key = max ? (long long)0x800fffffffffffffull : 0x7ff0000000000000ll;
    }
    __device__ void add(double x) {
        const long long b = __double_as_longlong(x), k = order(b);
        const bool nan = (b & 0x7fffffffffffffffll) > 0x7ff0000000000000ll;
        if (!nan && (max ? k > key : k < key)) key = k;
    }
    __device__ double get() const { return __longlong_as_double(order(key)); }
};
template <typename R> struct RedExtreme;
template <> struct RedExtreme<float> { using type = RedExtreme32; };
template <> struct RedExtreme<double> { using type = RedExtreme64; };

template <typename R> __device__ __forceinline__ bool red_nonfinite(R v);
template <> __device__ __forceinline__ bool red_nonfinite<double>(double v) {
    return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000;
}
template <> __device__ __forceinline__ bool red_nonfinite<float>(float v) {
    return (__float_as_int(v) & 0x7f800000) == 0x7f800000;
}

// Quantities of the cell alone: Q = the field pk.p[0], |u| or E_K.
enum { RED_FIELD, RED_UMAG, RED_EKIN };
template <typename R, int Q>
__global__ void __launch_bounds__(RED_THREADS) reduce_cells_kernel(PtrPack<const R> pk, Geom g, int op,
                                                                   double count, RedOut out) {
    __shared__ fx_u64 etab[Q == RED_EKIN && sizeof(R) == 8 ? 256 : 1];
    if (Q == RED_EKIN && sizeof(R) == 8) {
        etab[threadIdx.x] = EXP_FIX[threadIdx.x];
        __syncthreads();
    }
    const long long n = (long long)g.nx * g.ny * g.nz;
    const long long stride = (long long)gridDim.x * RED_THREADS;
    const bool extreme = op == AC_MAX || op == AC_MIN;
    typename RedExtreme<R>::type ext(op);
    double acc = 0.0;
    unsigned int bad = 0;
    constexpr int U = Q == RED_FIELD ? 8 : 4;  // cells in flight per thread
    for (long long t0 = blockIdx.x * (long long)RED_THREADS + threadIdx.x; t0 < n; t0 += U * stride) {
        R v[U][Q == RED_FIELD ? 1 : 4];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            long long o = t0 + u * stride < n ? t0 + u * stride : t0;
            if (g.padded) {
                const long long row = o / g.nx, i = o - row * g.nx, kz = row / g.ny;
                o = g.origin + kz * g.pxy + (row - kz * g.ny) * g.px + i;
            }
            if (Q == RED_FIELD) {
                v[u][0] = ldg(pk.p[0] + o);
            } else {
#pragma unroll
                for (int q = 0; q < (Q == RED_EKIN ? 4 : 3); ++q)
                    v[u][q] = ldg(pk.p[Q == RED_EKIN ? q : 1 + q] + o);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (t0 + u * stride >= n) break;
            R x = v[u][0];
            if (Q == RED_UMAG) x = v[u][0] * v[u][0] + v[u][1] * v[u][1] + v[u][2] * v[u][2];
            if (Q == RED_EKIN) {
                const R u2 = v[u][1] * v[u][1] + v[u][2] * v[u][2] + v[u][3] * v[u][3];
                if constexpr (sizeof(R) == 8) {
                    // |ln rho| < 64: the fixed-point exp
                    const bool in = (__double2hiint(x) & 0x7fffffff) < 0x40500000;
                    x = 0.5 * (in ? fx_exp55(fx_from_double55(x), etab, FX_L70) : exp(x)) * u2;
                } else {
                    x = (R)0.5 * exp(x) * u2;
                }
            }
            if (red_nonfinite(x)) bad = 1;
            if (extreme)
                ext.add(x);
            else if (Q == RED_UMAG && sizeof(R) == 8 && op == AC_RMS)  // |u|^2 itself
                acc += x;
            else if (Q == RED_UMAG) {
                const double v = sqrt(x);
                acc = op == AC_RMS ? fma(v, v, acc) : acc + v;
            }
            else
                acc = op == AC_RMS ? fma((double)x, (double)x, acc) : acc + (double)x;
        }
    }
    red_finish<R>(out, op, extreme ? ext.get() : acc, bad, count, extreme && Q == RED_UMAG);
}

// ---- quantities with B = curl A -----------------------------------------------------

// Tile t of a march: 32 x 8 columns, RED_Z planes.
constexpr int RED_Z = 16;
struct RedTile {
    int i, j, k0, k1;
    bool active;
    __device__ RedTile(long long t, const Geom &g) {
        const int gx = (g.nx + 31) / 32, gy = (g.ny + 7) / 8;
        const long long zt = t / ((long long)gx * gy);
        const int r = (int)(t - zt * gx * gy);
        i = (r % gx) * 32 + threadIdx.x;
        j = (r / gx) * 8 + threadIdx.y;
        k0 = (int)zt * RED_Z;
        k1 = min(k0 + RED_Z, g.nz);
        active = i < g.nx && j < g.ny;
    }
};
static long long red_tiles(const Geom &g) {
    return (long long)((g.nx + 31) / 32) * ((g.ny + 7) / 8) * ((g.nz + RED_Z - 1) / RED_Z);
}

// |B|^2 at a cell from integers; binary64 stencils where an exponent is out of range
// (non-finite values among them).  Each derivative has a scale of its own, the largest
// exponent among its six values: a uniform part of A, or another component's size, then
// takes no bits from it.  Values within three binades of that exponent are exact (a
// smaller one keeps the bits that a binary64 difference with the largest would keep, and
// three more), the numerator is their exact sum, rounded once to binary64.
template <class IX>
__device__ __forceinline__ double red_curl2(const double *const *f, const IX &ix,
                                            const DevCoefs<double> &k) {
    // derivative of A_q along axis a, d = 0..5 for the points -3 .. 3
    constexpr int Q[6] = {2, 1, 0, 2, 1, 0}, A[6] = {1, 2, 2, 0, 0, 1};
    double v[6][6];
#pragma unroll
    for (int t = 0; t < 6; ++t)
#pragma unroll
        for (int d = 0; d < 6; ++d) {
            const int m = d < 3 ? d - 3 : d - 2;
            v[t][d] = ldg(f[5 + Q[t]] + ix(A[t] == 0 ? m : 0, A[t] == 1 ? m : 0, A[t] == 2 ? m : 0));
        }
    int E[6];
    bool out = false;  // beyond 2^+-200
#pragma unroll
    for (int t = 0; t < 6; ++t) {
        int top = 0;
#pragma unroll
        for (int d = 0; d < 6; ++d) {
            const int h = __double2hiint(v[t][d]) & 0x7fffffff;
            top = h > top ? h : top;
        }
        E[t] = top >> 20;
        out |= E[t] >= 1223 || (E[t] < 823 && top > 0);
        E[t] = E[t] < 823 ? 823 : E[t];  // all zero
    }
    double B[3];
    if (out) {
        const GlobalView<double, IX> ax{f[5], ix}, ay{f[6], ix}, az{f[7], ix};
        B[0] = op_d1<1>(az, k.d1[1]) - op_d1<2>(ay, k.d1[2]);
        B[1] = op_d1<2>(ax, k.d1[2]) - op_d1<0>(az, k.d1[0]);
        B[2] = op_d1<0>(ay, k.d1[0]) - op_d1<1>(ax, k.d1[1]);
    } else {
        double d[6];
#pragma unroll
        for (int t = 0; t < 6; ++t) {
            long long F[6];
#pragma unroll
            for (int p = 0; p < 6; ++p) F[p] = fx_align(fx_double_to_bits(v[t][p]), E[t]);
            const long long n = 45 * (F[3] - F[2]) + 9 * (F[1] - F[4]) + (F[5] - F[0]);
            d[t] = fx_to_double(n, FX_EB64 + E[t] - 1078);
        }
        // (the weight of the outermost points is 1 / (60 dx))
#pragma unroll
        for (int q = 0; q < 3; ++q)
            B[q] = d[2 * q] * k.d1[A[2 * q]][2] - d[2 * q + 1] * k.d1[A[2 * q + 1]][2];
    }
    return B[0] * B[0] + B[1] * B[1] + B[2] * B[2];
}

// E_M (CFL = false), or the CFL speed of binary32 fields, over marching threads.
template <typename R, class IX, bool CFL>
__global__ void __launch_bounds__(RED_THREADS, 2)
    reduce_curl_kernel(PtrPack<const R> pk, Geom g, DevCoefs<R> k, int op, double count, long long tiles,
                       RedOut out) {
    double acc = red_init(op);
    unsigned int bad = 0;
    for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
        const RedTile c(t, g);
        if (!c.active) continue;
        IX ix;
        ix.set_xy(c.i, c.j, g);
        for (int z = c.k0; z < c.k1; ++z) {
            ix.set_z(z, g);
            double v;
            if constexpr (sizeof(R) == 8)
                v = 0.5 * red_curl2(pk.p, ix, k);
            else
                v = cell_quantity<R, IX>(pk.p, ix, k, CFL ? AC_Q_CFL : AC_Q_EMAG);
            if (red_nonfinite(v)) bad = 1;
            acc = red_combine(op, acc, op == AC_RMS ? v * v : v);
        }
    }
    red_finish<R>(out, op, acc, bad, count, false);
}

template <int A> struct RedAxis { static constexpr int value = A; };

// ---- the largest CFL speed of binary64 fields ------------------------------------------

// The exact speed of one cell folded into word (bits of a non-negative double).
template <class IX>
__device__ __forceinline__ void red_cfl_exact(const double *const *f, const IX &ix,
                                              const DevCoefs<double> &k, fx_u64 *word,
                                              unsigned int &bad) {
    const double v = cell_quantity<double, IX>(f, ix, k, AC_Q_CFL);
    if (red_nonfinite(v)) bad = 1;
    if (v == v) atomicMax(word, (fx_u64)__double_as_longlong(v));
}

// A block's non-finite cells noted in the flag word after the maximum.  Every kernel that
// takes exact speeds notes its own: once an infinity is in the word, later cells of the
// search compare against it.
__device__ __forceinline__ void red_cfl_flag(unsigned int bad, fx_u64 *word) {
    if (__syncthreads_or(bad) && threadIdx.x + threadIdx.y == 0)
        atomicOr(reinterpret_cast<unsigned int *>(word + 1), 1u);
}

// A first guess: the speeds of one cell in 8 x 8 x 4 (y, z, x).
template <class IX>
__global__ void __launch_bounds__(RED_THREADS) reduce_cfl_sample_kernel(PtrPack<const double> pk,
                                                                        Geom g, DevCoefs<double> k,
                                                                        fx_u64 *word) {
    const int nx = (g.nx + 3) / 4, ny = (g.ny + 7) / 8, nz = (g.nz + 7) / 8;
    const long long total = (long long)nx * ny * nz;
    unsigned int bad = 0;
    for (long long t = blockIdx.x * (long long)RED_THREADS + threadIdx.x; t < total;
         t += (long long)gridDim.x * RED_THREADS) {
        const long long r = t / nx;
        IX ix;
        ix.set_xy((int)(t - r * nx) * 4, (int)(r % ny) * 8, g);
        ix.set_z((int)(r / ny) * 8, g);
        red_cfl_exact(pk.p, ix, k, word, bad);
    }
    red_cfl_flag(bad, word);
}

// v in binary32 towards zero, but infinite or NaN, and |v| from 2^128 on, as infinity:
// a bound formed of such values is infinite or NaN.
__device__ __forceinline__ float red_float(double v) {
    const int hi = __double2hiint(v), a = hi & 0x7fffffff;
    int r = ((a - 0x38000000) << 3) | (int)((unsigned)__double2loint(v) >> 29);
    r = a < 0x38100000 ? 0 : (a >= 0x47f00000 ? 0x7f800000 : r);
    return __int_as_float(r | (hi & 0x80000000));
}

template <class IX>
__global__ void __launch_bounds__(RED_THREADS, 2)
    reduce_cfl_max_kernel(PtrPack<const double> pk, Geom g, DevCoefs<double> k, float3 c1, float cs2_ref,
                          float gamma_cp, float gm1, long long tiles, fx_u64 *word, RedOut out) {
    unsigned int bad = 0;
    const double *const *f = pk.p;
    for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
        const RedTile c(t, g);
        if (!c.active) continue;
        IX ix;
        ix.set_xy(c.i, c.j, g);
        for (int z = c.k0; z < c.k1; ++z) {
            ix.set_z(z, g);
            // derivatives of A in binary32, and s, the sum of the points' magnitudes
            float s = 0.f;
            auto d1 = [&](int q, auto axis) {
                constexpr int AX = decltype(axis)::value;
                float n = 0.f;
#pragma unroll
                for (int m = 1; m <= 3; ++m) {
                    const float w = m == 1 ? 45.f : (m == 2 ? -9.f : 1.f);
                    const float p = red_float(ldg(f[q] + ix(AX == 0 ? m : 0, AX == 1 ? m : 0, AX == 2 ? m : 0)));
                    const float n1 = red_float(ldg(f[q] + ix(AX == 0 ? -m : 0, AX == 1 ? -m : 0, AX == 2 ? -m : 0)));
                    s += fabsf(p) + fabsf(n1);
                    n = fmaf(w, p - n1, n);
                }
                return n * (AX == 0 ? c1.x : (AX == 1 ? c1.y : c1.z));
            };
            using X = RedAxis<0>;
            using Y = RedAxis<1>;
            using Z = RedAxis<2>;
            const float bx = d1(7, Y{}) - d1(6, Z{}), by = d1(5, Z{}) - d1(7, X{}),
                        bz = d1(6, X{}) - d1(5, Y{});
            // rounding of the values, differences and sums: below 2^-21 45 s a component
            const float e = s * (45.f * 0x1p-21f) * fmaxf(c1.x, fmaxf(c1.y, c1.z));
            const float Bx = fabsf(bx) + e, By = fabsf(by) + e, Bz = fabsf(bz) + e;
            const long long o = ix(0, 0, 0);
            const float ux = red_float(ldg(f[1] + o)), uy = red_float(ldg(f[2] + o)),
                        uz = red_float(ldg(f[3] + o));
            const float l = red_float(ldg(f[0] + o)), ss = red_float(ldg(f[4] + o));
            // e^x of a binary32 sum x: relative error below 2^-21 (1 + the terms' magnitudes)
            const float a = gamma_cp * ss, b = gm1 * l;
            const float grow = 1.0001f + 0x1p-20f * (fabsf(a) + fabsf(b) + fabsf(l));
            const float cs2 = cs2_ref * expf(a + b) * grow, ri = expf(-l) * grow;
            // (1e-37: what the squares lose below binary32's range)
            float up = 1.0001f * (sqrtf(ux * ux + uy * uy + uz * uz + 1e-37f) +
                                  sqrtf(cs2 + (Bx * Bx + By * By + Bz * Bz + 1e-37f) * ri));
            if (!(fabsf(a + b) <= 60.f && fabsf(l) <= 60.f)) up = INFINITY;
            // (at most binary32's largest number: an infinite bound is never below it, and
            // the cell's exact speed is taken, however large the known one)
            const float known = fminf(red_float(__longlong_as_double((long long)*
                                      reinterpret_cast<volatile fx_u64 *>(word))), FLT_MAX);
            if (!(up <= known)) red_cfl_exact(f, ix, k, word, bad);
        }
    }
    red_cfl_flag(bad, word);
    if (red_last_block(out.flags + RED_MAX_BLOCKS) && threadIdx.x + threadIdx.y == 0) {
        const fx_u64 w = __ldcg(word);
        const unsigned int b = __ldcg(reinterpret_cast<unsigned int *>(word + 1));
        red_write(out, b && w == 0 ? -INFINITY : __longlong_as_double((long long)w), b);
    }
}

template <class IX>
static cudaError_t launch_cfl_max(const ReduceLaunch &L, const PtrPack<const double> &pk,
                                  const DevCoefs<double> &k, const RedOut &out, unsigned nb,
                                  long long tiles, cudaStream_t st, int *launches) {
    fx_u64 *word = reinterpret_cast<fx_u64 *>(L.partials);  // max, then the flag word
    cudaError_t e = cudaMemsetAsync(word, 0, 2 * sizeof(fx_u64), st);
    if (e != cudaSuccess) return e;
    if ((long long)L.g.nx * L.g.ny * L.g.nz >= 1 << 16) {
        const long long n = (long long)((L.g.nx + 3) / 4) * ((L.g.ny + 7) / 8) * ((L.g.nz + 7) / 8);
        const long long b = (n + RED_THREADS - 1) / RED_THREADS;
        reduce_cfl_sample_kernel<IX><<<(unsigned)(b < 1216 ? b : 1216), RED_THREADS, 0, st>>>(pk, L.g, k, word);
        ++*launches;
    }
    const float3 c1 = make_float3((float)L.c.d1[0][2], (float)L.c.d1[1][2], (float)L.c.d1[2][2]);
    reduce_cfl_max_kernel<IX><<<nb, dim3(32, 8), 0, st>>>(pk, L.g, k, c1, (float)L.ph.cs2_ref,
                                                          (float)L.ph.gamma_cp, (float)L.ph.gm1, tiles,
                                                          word, out);
    ++*launches;
    return cudaGetLastError();
}

// B = curl A at the sixth order; false where the general kernel has to do it.
template <typename R, class IX>
static bool launch_curl(const ReduceLaunch &L, const PtrPack<const R> &pk, const DevCoefs<R> &k,
                        const RedOut &out, double count, cudaStream_t st, int *launches,
                        cudaError_t *err) {
    const long long tiles = red_tiles(L.g);
    const unsigned nb = (unsigned)(tiles < RED_MAX_BLOCKS ? tiles : RED_MAX_BLOCKS);
    const bool sum = L.op == AC_SUM || L.op == AC_RMS;
    if (L.quantity == AC_Q_EMAG) {
        if (!sum) return false;
        reduce_curl_kernel<R, IX, false><<<nb, dim3(32, 8), 0, st>>>(pk, L.g, k, L.op, count, tiles, out);
        ++*launches;
        *err = cudaGetLastError();
        return true;
    }
    if constexpr (sizeof(R) == 8) {
        // (the binary32 bound wants c_s and the spacings of ordinary magnitude)
        const double lo = fmin(L.dx[0], fmin(L.dx[1], L.dx[2])), hi = fmax(L.dx[0], fmax(L.dx[1], L.dx[2]));
        if (L.op != AC_MAX || !(L.ph.cs2_ref >= 1e-10 && L.ph.cs2_ref <= 1e10) || !(hi <= 8.0 * lo) ||
            !(lo >= 1e-12 && hi <= 1e12))
            return false;
        *err = launch_cfl_max<IX>(L, pk, k, out, nb, tiles, st, launches);
    } else {
        reduce_curl_kernel<R, IX, true><<<nb, dim3(32, 8), 0, st>>>(pk, L.g, k, L.op, count, tiles, out);
        ++*launches;
        *err = cudaGetLastError();
    }
    return true;
}

template <typename R>
static cudaError_t launch_reduce_t(const ReduceLaunch &L, cudaStream_t st, int *launches) {
    PtrPack<const R> pk;
    for (int q = 0; q < NF; ++q) pk.p[q] = static_cast<const R *>(L.f[q]);
    const DevCoefs<R> k = to_dev<R>(L.c, L.ph);
    const long long total = (long long)L.g.nx * L.g.ny * L.g.nz;
    const long long rows = (long long)L.g.ny * L.g.nz;
    const RedOut out{L.partials, L.flags, L.result, L.host};
    const double count = (double)total;
    const bool sum = L.op == AC_SUM || L.op == AC_RMS;
    if (L.quantity <= AC_Q_UMAG || (L.quantity == AC_Q_EKIN && sum)) {
        long long b = (total + 4 * RED_THREADS - 1) / (4 * RED_THREADS);
        const unsigned nb = (unsigned)(b < 1 ? 1 : (b > L.blocks ? L.blocks : b));
        if (L.quantity < NF) {
            pk.p[0] = pk.p[L.quantity];
            reduce_cells_kernel<R, RED_FIELD><<<nb, RED_THREADS, 0, st>>>(pk, L.g, L.op, count, out);
        } else if (L.quantity == AC_Q_UMAG) {
            reduce_cells_kernel<R, RED_UMAG><<<nb, RED_THREADS, 0, st>>>(pk, L.g, L.op, count, out);
        } else {
            reduce_cells_kernel<R, RED_EKIN><<<nb, RED_THREADS, 0, st>>>(pk, L.g, L.op, count, out);
        }
        ++*launches;
        return cudaGetLastError();
    }
    if (L.c.radius == 3 && L.quantity >= AC_Q_EMAG) {
        cudaError_t e = cudaSuccess;
        const bool done =
            L.g.padded ? launch_curl<R, IdxPadded>(L, pk, k, out, count, st, launches, &e)
            : L.g.elems < (1ll << 31)
                ? launch_curl<R, IdxPeriodic32>(L, pk, k, out, count, st, launches, &e)
                : launch_curl<R, IdxPeriodic>(L, pk, k, out, count, st, launches, &e);
        if (done) return e;
    }
    long long blocks = (rows + RED_THREADS / 32 - 1) / (RED_THREADS / 32);
    if (blocks > L.blocks) blocks = L.blocks;
    if (blocks < 1) blocks = 1;
    const unsigned nb = (unsigned)blocks;
#define AC_RED(IX, RAD) \
    reduce_kernel<R, IX, RAD><<<nb, RED_THREADS, 0, st>>>(pk, L.g, k, L.op, L.quantity, count, out)
    // B = curl A uses the handle's stencil order (padded layout: radius <= 3)
    switch (L.c.radius) {
        case 1: if (L.g.padded) AC_RED(IdxPadded, 1); else AC_RED(IdxPeriodicR<1>, 1); break;
        case 2: if (L.g.padded) AC_RED(IdxPadded, 2); else AC_RED(IdxPeriodicR<2>, 2); break;
        case 4: AC_RED(IdxPeriodicR<4>, 4); break;
        default: if (L.g.padded) AC_RED(IdxPadded, 3); else AC_RED(IdxPeriodic, 3); break;
    }
#undef AC_RED
    ++*launches;
    return cudaGetLastError();
}

cudaError_t launch_reduce(const ReduceLaunch &L, cudaStream_t st, int *launches) {
    if (L.precision == AC_FP64) return launch_reduce_t<double>(L, st, launches);
    return launch_reduce_t<float>(L, st, launches);
}

}  // namespace ac

#ifdef AC_BOUNDS_CHECK
namespace ac {
// Self-test of the checks: two indices are only computed, never used to
// address memory: -5 against an extent of 10 must be recorded (tag 7) and
// redirected to 0, 3 must pass unchanged.
__global__ void bc_selftest_kernel(long long *out) {
    out[0] = AC_BC(-5ll, 10ll, 7u);
    out[1] = AC_BC(3ll, 10ll, 7u);
}
}  // namespace ac
#endif

extern "C" int ac_bounds_check_selftest(long long out[2]) {
    if (!out) return AC_ERR_ARG;
#ifdef AC_BOUNDS_CHECK
    long long *d = nullptr;
    cudaError_t e = cudaMalloc(&d, 2 * sizeof(long long));
    if (e == cudaSuccess) {
        ac::bc_selftest_kernel<<<1, 1>>>(d);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(out, d, 2 * sizeof(long long), cudaMemcpyDeviceToHost);
    if (d) cudaFree(d);
    return e == cudaSuccess ? AC_OK : ac::ac_report_cuda(e);
#else
    out[0] = out[1] = 0;
    return AC_ERR_STATE;
#endif
}

AC_BC_READER(bc_take_aux)
