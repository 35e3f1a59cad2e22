// k_util.cu -- set-up and data-movement kernels of libbgk: sampling the initial Maxwellian into the
// device layout, and converting f between the host order [point][velocity] (FP64) and the device
// tile layout f[vt][e][i][lane] (FP32).
#include <algorithm>

#include "bgk_common.cuh"

namespace bgk {

// Sample the continuous Maxwellian (Sec. 2, Eq. 4, velocity dimension m = 3, or 2 when nz = 1: the
// one z node has factor 1 and U_z takes no part) of every point's primitive state into f. A CTA owns PB
// consecutive points (of as many elements as that takes) and a run of velocity tiles: the separable
// factors exp(-(xi_d - U_d)^2 / (2 theta)) of its points are tabulated once in shared memory as FP32 (the
// exponent in FP64, split into an integer power of two and a remainder in [-1/2, 1/2] whose 2^r is taken
// in FP32: within a few FP32 ulp at any exponent), then every (tile, point, lane) value is the product
// (C Ex) Ey Ez. Writes 0 on padded slots.
// Q (when not null): the discrete moments (Eq. 2 with Eq. 12) of every point's sampled Maxwellian in
// FP64, from the 1-D trapezoid sums of its tabulated factors (the grid is a tensor product): they differ
// from the moments of the stored FP32 values only by the rounding of the products.
// Bound: the tables by the FP64 pipe (a warp instruction per 16 clocks, whatever its active lanes), the
// values by the writing of f. One CTA per element left most lanes of the table and moment work idle at
// four points per element, and a small mesh's tiles to a few CTAs. 65,536 line elements at p = 3, 32^2
// velocities (1.1 GB of f): 3.24 ms before, 0.61 now; 128^2 quadrilaterals 1.37 -> 0.61; 16^3
// hexahedra, 24^3 velocities (14.5 GB) 3.34 -> 2.02.
// (n = rint(y) by the rounding constant 1.5 2^52, whose low word then holds n: two FP64 operations for three
// and a conversion. Below 2^-2000 the result is 0 anyway and n would not fit.)
__device__ __forceinline__ float exp_split(double x)
{
    const double y = x * 1.4426950408889634;  // log2(e); y <= 0
    if ((unsigned)__double2hiint(y) > 0xc09f4000u)  // y < -2000, or NaN
        return y < 0.0 ? 0.f : (float)y;
    const double t = __dadd_rn(y, 6755399441055744.0);
    const double n = __dsub_rn(t, 6755399441055744.0);
    return ldexpf(exp2f((float)(y - n)), __double2loint(t));
}
// the exact double of a non-negative FP32 value without the FP64 pipe's conversion
__device__ __forceinline__ double widen(float v)
{
    const unsigned u = __float_as_uint(v);
    if (u - 0x00800000u >= 0x7f000000u)  // zero, subnormal, infinite or NaN
        return (double)v;
    return __hiloint2double((int)((u >> 3) + 0x38000000u), (int)(u << 29));
}

__global__ void __launch_bounds__(256, 4)
    k_init_maxwellian(float *__restrict__ f, const double *__restrict__ prim, const float *__restrict__ mi,
                      const float *__restrict__ gmask, int nslots, int nvt, int npts, int PB, int tiles, int nx, int ny,
                      int nz, double v0x, double v0y, double v0z, double dvx, double dvy, double dvz, int *err,
                      double *__restrict__ Q, double *__restrict__ warm)
{
    const double hm = nz == 1 ? 1.0 : 1.5;  // m / 2
    const int ntab = nx + ny + nz + 1;       // per point: 0 (padded slots), then the factors by axis
    extern __shared__ double ith[];          // [PB] -1 / (2 theta) of the CTA's points,
    double *S = ith + PB;                    // [PB][3][3] 1-D sums,
    double *xg = S + 9 * PB;                 // [ntab - 1] velocities of the nodes, axis by axis,
    double *x2 = xg + (ntab - 1);            // [ntab - 1] and their squares,
    float *cn = reinterpret_cast<float *>(x2 + (ntab - 1));  // [PB] normalisations,
    float *tab = cn + PB;                    // [PB][ntab]
    const int p0 = blockIdx.x * PB, np = min(PB, npts - p0);
    const bool first = blockIdx.y == 0;      // writes the points' moments and warm starts
    // per point: the normalisation rho (2 pi theta)^(-m/2) and -1 / (2 theta) (one division per point)
    for (int i = threadIdx.x; i < np; i += blockDim.x) {
        const double *s = prim + (int64_t)(p0 + i) * 5;
        const double rho = s[0], th = s[4];
        const bool ok = rho > 0.0 && th > 0.0;
        if (!ok)
            atomicOr(err, kErrDomain);
        ith[i] = ok ? -0.5 / th : 0.0;
        const double C = rho * pow(2.0 * 3.14159265358979323846 * th, -hm);
        cn[i] = ok ? (float)C : 0.f;
        tab[i * ntab] = 0.f;
        if (warm && ok && first) {  // the first Newton solve's start: this Maxwellian, (ln C, U, theta)
            double *wp = warm + (int64_t)(p0 + i) * 5;
            wp[0] = log(C);
            wp[1] = s[1];
            wp[2] = s[2];
            wp[3] = nz == 1 ? 0.0 : s[3];
            wp[4] = th;
        }
    }
    for (int t = threadIdx.x; t < ntab - 1; t += blockDim.x) {
        const int d = t < nx ? 0 : (t < nx + ny ? 1 : 2), k = t - (d > 0 ? nx : 0) - (d > 1 ? ny : 0);
        xg[t] = fma((double)k, d == 0 ? dvx : (d == 1 ? dvy : dvz), d == 0 ? v0x : (d == 1 ? v0y : v0z));
        x2[t] = xg[t] * xg[t];
    }
    __syncthreads();
    for (int q = threadIdx.x; q < np * (ntab - 1); q += blockDim.x) {
        const int i = q / (ntab - 1), t = q % (ntab - 1);
        const double a = ith[i];
        float v = 1.f;
        if (t < nx + ny || nz > 1) {
            const double c = xg[t] - prim[(int64_t)(p0 + i) * 5 + (t < nx ? 1 : (t < nx + ny ? 2 : 3))];
            v = exp_split(a * c * c);
        }
        tab[i * ntab + 1 + t] = a == 0.0 ? 0.f : v;
    }
    __syncthreads();
    if (Q && first) {
        // the 1-D sums of every (point, axis) by a thread of its own, then the points' moments
        for (int q = threadIdx.x; q < 3 * np; q += blockDim.x) {
            const int d = q / np, i = q % np;
            const int n = d == 0 ? nx : (d == 1 ? ny : nz);
            const double dv = d == 0 ? dvx : (d == 1 ? dvy : dvz), hv = 0.5 * dv;
            const int o = (d > 0 ? nx : 0) + (d > 1 ? ny : 0);
            const float *t = tab + i * ntab + 1 + o;
            double s0 = 0.0, s1 = 0.0, s2 = 0.0;
            if (n == 1) {  // the absent u_z: one node at 0 of unit weight
                s0 = (double)t[0];
            } else {
                for (int k = 0; k < n; k++) {
                    const double a = (k == 0 || k == n - 1 ? hv : dv) * widen(t[k]);
                    s0 += a;
                    s1 = fma(xg[o + k], a, s1);
                    s2 = fma(x2[o + k], a, s2);
                }
            }
            double *so = S + (i * 3 + d) * 3;
            so[0] = s0;
            so[1] = s1;
            so[2] = s2;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < np; i += blockDim.x) {
            const double(*s)[3] = reinterpret_cast<const double(*)[3]>(S + 9 * i);
            const double C = (double)cn[i];
            double *q = Q + (int64_t)(p0 + i) * 5;
            q[0] = C * s[0][0] * s[1][0] * s[2][0];
            q[1] = C * s[0][1] * s[1][0] * s[2][0];
            q[2] = C * s[0][0] * s[1][1] * s[2][0];
            q[3] = C * s[0][0] * s[1][0] * s[2][1];
            q[4] = 0.5 * C * (s[0][2] * s[1][0] * s[2][0] + s[0][0] * s[1][2] * s[2][0] + s[0][0] * s[1][0] * s[2][2]);
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < np * nx; q += blockDim.x)  // the normalisation into the x factors
        tab[(q / nx) * ntab + 1 + q % nx] *= cn[q / nx];
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    // the tile's table columns (1 + k_x, 1 + n_x + k_y, 1 + n_x + n_y + k_z) from the centred index table
    // (k_d = (m_d + n_d - 1) / 2, exact), column 0 on padded slots; the warp's next tile's are loaded while
    // this one is written
    auto slot_cols = [&](int vt, int &cx, int &cy, int &cz) {
        const int slot = vt * kWarp + lane;
        cx = 1 + __float2int_rn(0.5f * (__ldg(mi + slot) + (float)(nx - 1)));
        cy = 1 + nx + __float2int_rn(0.5f * (__ldg(mi + nslots + slot) + (float)(ny - 1)));
        cz = 1 + nx + ny + __float2int_rn(0.5f * (__ldg(mi + 2 * nslots + slot) + (float)(nz - 1)));
        if (__ldg(gmask + slot) == 0.f)
            cx = 0;
    };
    // a warp per tile, all of the CTA's points: the tile's columns are loaded once and serve PB rows
    const int vt1 = min((int)(blockIdx.y + 1) * tiles, nvt);
    int vt = blockIdx.y * tiles + w;
    if (vt >= vt1)
        return;
    int cx, cy, cz;
    slot_cols(vt, cx, cy, cz);
    for (; vt < vt1; vt += nw) {
        int nx_ = 0, ny_ = 0, nz_ = 0;
        if (vt + nw < vt1)
            slot_cols(vt + nw, nx_, ny_, nz_);
        float *dst = f + ((int64_t)vt * npts + p0) * kWarp + lane;
        const float *tx = tab + cx, *ty = tab + cy, *tz = tab + cz;
#pragma unroll 8
        for (int i = 0; i < np; i++)
            __stcs(dst + i * kWarp, tx[i * ntab] * ty[i * ntab] * tz[i * ntab]);
        cx = nx_;
        cy = ny_;
        cz = nz_;
    }
}

// f (device tiles, FP32) <- host-order staging [pt - p0][k] (FP64) for points [p0, p0 + npt)
__global__ void k_scatter_f(float *__restrict__ f, const double *__restrict__ st, const int *__restrict__ slotk,
                            int nvt, int E, int NP, int64_t nvel, int p0, int npt)
{
    const int64_t n = (int64_t)nvt * npt * kWarp;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const int lane = (int)(q % kWarp);
        const int pl = (int)((q / kWarp) % npt);
        const int vt = (int)(q / ((int64_t)kWarp * npt));
        const int k = __ldg(slotk + vt * kWarp + lane);
        const int pt = p0 + pl;
        f[fidx(vt, pt / NP, pt % NP, lane, E, NP)] = k < 0 ? 0.f : (float)st[(int64_t)pl * nvel + k];
    }
}

// host-order staging [pt - p0][k] (FP64) <- f (device tiles)
__global__ void k_gather_f(double *__restrict__ st, const float *__restrict__ f, const int *__restrict__ slotk,
                           int nvt, int E, int NP, int64_t nvel, int p0, int npt)
{
    const int64_t n = (int64_t)nvt * npt * kWarp;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const int lane = (int)(q % kWarp);
        const int pl = (int)((q / kWarp) % npt);
        const int vt = (int)(q / ((int64_t)kWarp * npt));
        const int k = __ldg(slotk + vt * kWarp + lane);
        if (k < 0)
            continue;
        const int pt = p0 + pl;
        st[(int64_t)pl * nvel + k] = (double)f[fidx(vt, pt / NP, pt % NP, lane, E, NP)];
    }
}

cudaError_t launch_init_maxwellian(float *f, const double *prim, const float *mi, const float *gmask, int nslots,
                                   int nvt, int E, int NP, const int n[3], const double v0[3], const double dv[3],
                                   int *err, double *Q, double *warm, cudaStream_t s)
{
    const int npts = E * NP, ntab = n[0] + n[1] + n[2] + 1;
    // points per CTA: 64, so that two warps of them fill the lanes of the FP64 work, but 32 where that leaves
    // fewer than two CTAs per SM, and no more than 96 KB of tables (two CTAs per SM) where the grid allows
    const int per = 10 * (int)sizeof(double) + (ntab + 1) * (int)sizeof(float);
    const int grid = 2 * (ntab - 1) * (int)sizeof(double);
    int PB = npts >= 64 * 304 ? 64 : 32;
    PB = std::max(1, std::min(PB, (98304 - grid) / per));
    const int smem = PB * per + grid;
    // runs of at least 32 tiles (their writing outweighs the tables that every run forms anew), as many as
    // two CTAs per SM take
    const int nb = (npts + PB - 1) / PB;
    const int runs = std::max(1, std::min((nvt + 31) / 32, 304 / nb));
    const int tiles = (nvt + runs - 1) / runs;
    cudaError_t e = cudaFuncSetAttribute(k_init_maxwellian, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess)
        return e;
    k_init_maxwellian<<<dim3(nb, (nvt + tiles - 1) / tiles), 256, smem, s>>>(
        f, prim, mi, gmask, nslots, nvt, npts, PB, tiles, n[0], n[1], n[2], v0[0], v0[1], v0[2], dv[0], dv[1], dv[2], err, Q,
        warm);
    return cudaGetLastError();
}

// Largest |a - b| and |b| over the real slots of two distributions stored in the same tile layout
// (each FP32 or FP64): out[0], out[1] hold the bit patterns of the two non-negative doubles, which
// order like the unsigned integers (atomicMax).
template <typename TA, typename TB>
__global__ void __launch_bounds__(256) k_f_distance(const TA *__restrict__ a, const TB *__restrict__ b,
                                                    const int *__restrict__ slotk, int64_t n, int per_tile,
                                                    unsigned long long *out)
{
    double d = 0.0, m = 0.0;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const int lane = (int)(q % kWarp);
        const int vt = (int)(q / per_tile);
        if (__ldg(slotk + vt * kWarp + lane) < 0)
            continue;
        const double x = (double)a[q], y = (double)b[q];
        d = fmax(d, fabs(x - y));
        m = fmax(m, fabs(y));
    }
    for (int o = 16; o > 0; o >>= 1) {
        d = fmax(d, __shfl_xor_sync(0xffffffffu, d, o));
        m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(out, (unsigned long long)__double_as_longlong(d));
        atomicMax(out + 1, (unsigned long long)__double_as_longlong(m));
    }
}

cudaError_t launch_f_distance(const void *a, bool a64, const void *b, bool b64, const int *slotk, int nvt, int E,
                              int NP, unsigned long long *out, cudaStream_t s)
{
    const int64_t n = (int64_t)nvt * E * NP * kWarp;
    const int per_tile = E * NP * kWarp;
    const int threads = 256;
    const int blocks = (int)std::min<int64_t>((n + threads - 1) / threads, 152 * 16);
    cudaError_t e = cudaMemsetAsync(out, 0, 2 * sizeof(unsigned long long), s);
    if (e != cudaSuccess)
        return e;
    if (a64 && b64)
        k_f_distance<<<blocks, threads, 0, s>>>((const double *)a, (const double *)b, slotk, n, per_tile, out);
    else if (a64)
        k_f_distance<<<blocks, threads, 0, s>>>((const double *)a, (const float *)b, slotk, n, per_tile, out);
    else if (b64)
        k_f_distance<<<blocks, threads, 0, s>>>((const float *)a, (const double *)b, slotk, n, per_tile, out);
    else
        k_f_distance<<<blocks, threads, 0, s>>>((const float *)a, (const float *)b, slotk, n, per_tile, out);
    return cudaGetLastError();
}

cudaError_t launch_convert_f(bool to_device, float *f, double *st, const int *slotk, int nvt, int E, int NP,
                             int64_t nvel, int p0, int npt, cudaStream_t s)
{
    const int64_t n = (int64_t)nvt * npt * kWarp;
    const int threads = 256;
    const int blocks = (int)std::min<int64_t>((n + threads - 1) / threads, 152 * 64);
    if (to_device)
        k_scatter_f<<<blocks, threads, 0, s>>>(f, st, slotk, nvt, E, NP, nvel, p0, npt);
    else
        k_gather_f<<<blocks, threads, 0, s>>>(st, f, slotk, nvt, E, NP, nvel, p0, npt);
    return cudaGetLastError();
}

}  // namespace bgk
