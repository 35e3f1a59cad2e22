// k_plain64.cu -- the plain all-FP64 form of the stage: f stored and advected in FP64, unfused.
//
// Per stage, k64_table tabulates the 1-D factors of every point's conservative Maxwellian (Sec. 2, Eq. 4;
// on the tensor velocity grid g = (C E_x[kx]) E_y[ky] E_z[kz]). Per velocity chunk k64_stage then forms
// the FR derivative with the upwind flux (Sec. 2.1, Eqs. 7-9) line by line and combines the relaxation
// and the Shu-Osher stage (k64_stage_curved on mapped elements). k64_moments sums the FP64 moments of the
// stage output over all chunks (warp per point), and the shared Newton kernel solves for the next
// Maxwellian from those FP64 moments. It is the straightforward comparison form: no fusion of stage and
// moments, no FP32, no staging by bulk copies.
// Everything here is bound by the FP64 pipe (2 operations per clock and SM, 1/64 of FP32's rate): what
// counts is the number of FP64 operations per degree of freedom, and loads and index arithmetic are free.
#include <algorithm>

#include "bgk_common.cuh"

namespace bgk {

// The exterior trace at face (d, side) of element e for the face point fp of the line whose own first
// node is i0 (stride along d): the neighbour's interpolant at the shared face (structured grid or the
// connectivity table), or the face's ghost (times the wall density on a diffuse wall).
__device__ double exterior64(const Stage64Args &A, int vl, int e, const int ec[3], int d, int side, int fp, int i0,
                             int lane, int slot)
{
    const int N1 = A.N1, NQ = N1 * N1, E = A.mesh.nelem, NP = A.NP;
    const int stride = d == 0 ? 1 : (d == 1 ? N1 : NQ);
    int en, g, base, str, wall = -1;
    bool hi;  // the neighbour's shared face is its +1 end
    if (A.ftab) {
        const int4 t = A.ftab[(int64_t)e * 6 + 2 * d + side];
        en = t.x;
        g = -1 - t.x;
        str = t.y;
        hi = t.z != 0;
        wall = t.w;
        base = A.fbase[((int64_t)e * 6 + 2 * d + side) * NQ + fp];
    } else {
        int nc[3] = {ec[0], ec[1], ec[2]};
        nc[d] += side ? 1 : -1;
        g = 2 * d + side;
        en = -1;
        if (nc[d] < 0 || nc[d] >= A.mesh.ne[d]) {
            if (A.mesh.bc[g] == 0)
                nc[d] = (nc[d] + A.mesh.ne[d]) % A.mesh.ne[d];
        }
        if (nc[d] >= 0 && nc[d] < A.mesh.ne[d])
            en = nc[0] + A.mesh.ne[0] * (nc[1] + A.mesh.ne[1] * nc[2]);
        str = stride;
        hi = side == 0;
        base = i0;
    }
    if (en < 0) {
        double up = A.ghost[(int64_t)g * A.nslots + slot];
        if (A.ftab) {
            if (wall >= 0)  // a wall face of the unstructured mesh
                up *= A.rhowu[(int64_t)wall * NQ + fp];
        } else if (A.mesh.bc[g] == 2) {
            up *= A.rhow[((int64_t)g * A.nfmax + face_elem(A.mesh, ec, d)) * NQ + fp];
        }
        return up;
    }
    double t = 0.0;
    for (int j = 0; j < N1; j++)
        t += (hi ? A.ops.lp[j] : A.ops.lm[j]) * A.src[fidx(vl, en, base + j * str, lane, E, NP)];
    return t;
}

// Curvilinear residual of one degree of freedom (node i of element e, one velocity): per direction the
// nodal fluxes F_j = (Ja^d(node_j) . xi) f_j along the line, D F, and the FR corrections with the upwind
// common fluxes of the shared face normals at both ends; -(sum over directions) / J.
__device__ double curved_residual64(const Stage64Args &A, int vl, int e, int i, int lane, int slot, const int ec[3],
                                    const int ic[3], const double xi[3])
{
    const int N1 = A.N1, NQ = N1 * N1, E = A.mesh.nelem, NP = A.NP;
    double R = 0.0;
    for (int d = 0; d < 3; d++) {
        const int stride = d == 0 ? 1 : (d == 1 ? N1 : NQ);
        const int i0 = i - ic[d] * stride;
        const int o1 = d == 0 ? 1 : 0, o2 = d == 2 ? 1 : 2;
        const int fp = ic[o1] + N1 * ic[o2];
        double dsum = 0.0, FL = 0.0, FR = 0.0, fL = 0.0, fR = 0.0;
        for (int j = 0; j < N1; j++) {
            const int node = i0 + j * stride;
            const double *ja = A.ja + (((int64_t)e * NP + node) * 3 + d) * 3;
            const double fj = A.src[fidx(vl, e, node, lane, E, NP)];
            const double Fj = (ja[0] * xi[0] + ja[1] * xi[1] + ja[2] * xi[2]) * fj;
            dsum += A.ops.D[ic[d]][j] * Fj;
            FL += A.ops.lm[j] * Fj;
            FR += A.ops.lp[j] * Fj;
            fL += A.ops.lm[j] * fj;
            fR += A.ops.lp[j] * fj;
        }
        const double *nL = A.fnm + ((((int64_t)e * 3 + d) * 2 + 0) * NQ + fp) * 3;
        const double *nR = A.fnm + ((((int64_t)e * 3 + d) * 2 + 1) * NQ + fp) * 3;
        const double uL = nL[0] * xi[0] + nL[1] * xi[1] + nL[2] * xi[2];
        const double uR = nR[0] * xi[0] + nR[1] * xi[1] + nR[2] * xi[2];
        const double FIL = uL > 0.0 ? uL * exterior64(A, vl, e, ec, d, 0, fp, i0, lane, slot) : uL * fL;
        const double FIR = uR < 0.0 ? uR * exterior64(A, vl, e, ec, d, 1, fp, i0, lane, slot) : uR * fR;
        R -= dsum + (FIL - FL) * A.ops.gl[ic[d]] + (FIR - FR) * A.ops.gr[ic[d]];
    }
    return R * A.ijac[(int64_t)e * NP + i];
}

// The 1-D factors of every point's Maxwellian, tab[n_x][n_x-axis + n_y + n_z]: E_d[k] =
// exp(-(xi_k - U_d)^2 / (2 theta)), the x factors with the normalisation C, from par = (C, U', 1/(2 theta')).
// 3 n exponentials per point instead of n^3.
__global__ void __launch_bounds__(256) k64_table(double *tab, const double *par, const Table64Args T, int npts)
{
    const int nt = T.n[0] + T.n[1] + T.n[2];
    const int64_t n = (int64_t)npts * nt;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t pt = q / nt;
        int k = (int)(q % nt), d = 0;
        if (k >= T.n[0])
            k -= T.n[d++];
        if (d == 1 && k >= T.n[1])
            k -= T.n[d++];
        const double *p = par + pt * 5;
        const double c = T.v0[d] + k * T.dv[d] - p[1 + d];
        tab[q] = (d == 0 ? p[0] : 1.0) * exp(-c * c * p[4]);
    }
}

// table columns of a slot's velocity
__device__ __forceinline__ void columns64(const Table64Args &T, int slot, int (&col)[3])
{
    int off = 0;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        col[d] = off + __float2int_rn(0.5f * (__ldg(T.mi + d * T.nslots + slot) + (float)(T.n[d] - 1)));
        off += T.n[d];
    }
}

// One warp per (velocity tile, element), lane = velocity: the FR derivative line by line, every line's sums
// shared by its nodes (s_i = sum_j DL_ij f_j + gl_i t_up with the interior trace folded into DL), the
// accumulators in the warp's shared memory, then the relaxation. FP64 operations per degree of freedom at
// p = 3 in 3-D: 27 (7 per direction, 3 for the Maxwellian, 3 to combine) against some 100 for one thread per
// degree of freedom with its own traces and an exponential. 6^3 elements at p = 3, 16^3 velocities:
// 1.58 -> 0.39 ms per chunk launch (the FP64 pipe's share of that: 0.33).
template <int N1>
__global__ void __launch_bounds__(kWarp) k64_stage(const Stage64Args A)
{
    extern __shared__ double acc64[];  // [NP][32]
    const int NP = A.NP, E = A.mesh.nelem, dim = A.mesh.dim, lane = threadIdx.x;
    const int vl = blockIdx.x / A.ecount, el = blockIdx.x % A.ecount, e = A.e0 + el;
    const int slot = (A.vt0 + vl) * kWarp + lane;
    const int ec[3] = {e % A.mesh.ne[0], (e / A.mesh.ne[0]) % A.mesh.ne[1], e / (A.mesh.ne[0] * A.mesh.ne[1])};
    const int oct = A.toct[A.vt0 + vl];
    double *acc = acc64 + lane;
    const double *fs = A.src + fidx(vl, e, 0, lane, E, NP);
    const double *fn = A.fn ? A.fn + fidx(vl, e, 0, lane, E, NP) : nullptr;
    for (int d = 0; d < dim; d++) {
        const double a = A.xi[d * A.nslots + slot];
        const bool left = (oct >> d) & 1;
        const double cd = -(2.0 / A.h[d]) * A.b * A.dt * a;
        const int stride = d == 0 ? 1 : (d == 1 ? N1 : N1 * N1), other = d == 0 ? N1 : 1, outer = d == 2 ? N1 : N1 * N1;
        // upwind neighbour (periodic wrap), or the ghost value of a boundary face (times the density of the
        // face point on a diffuse wall)
        int nc[3] = {ec[0], ec[1], ec[2]};
        nc[d] += left ? -1 : 1;
        const double *up = nullptr, *rw = nullptr;
        double gh = 0.0;
        const int fc = 2 * d + (left ? 0 : 1);
        if ((nc[d] < 0 || nc[d] >= A.mesh.ne[d]) && A.mesh.bc[fc] != 0) {
            gh = A.ghost[fc * A.nslots + slot];
            if (A.mesh.bc[fc] == 2)
                rw = A.rhow + ((int64_t)fc * A.nfmax + face_elem(A.mesh, ec, d)) * N1 * N1;
        } else {
            nc[d] = (nc[d] + A.mesh.ne[d]) % A.mesh.ne[d];
            up = A.src + fidx(vl, nc[0] + A.mesh.ne[0] * (nc[1] + A.mesh.ne[1] * nc[2]), 0, lane, E, NP);
        }
        for (int ln = 0; ln < NP / N1; ln++) {  // ln: the line's face point
            const int i0 = (ln % N1) * other + (ln / N1) * outer;
            double f[N1], t = gh;
#pragma unroll
            for (int j = 0; j < N1; j++)
                f[j] = fs[(i0 + j * stride) * kWarp];
            if (up) {
                t = 0.0;
#pragma unroll
                for (int j = 0; j < N1; j++)
                    t = fma(left ? A.ops.lp[j] : A.ops.lm[j], up[(i0 + j * stride) * kWarp], t);
            } else if (rw) {
                t *= rw[ln];
            }
#pragma unroll
            for (int i = 0; i < N1; i++) {
                double v = (left ? A.ops.gl[i] : A.ops.gr[i]) * t;
#pragma unroll
                for (int j = 0; j < N1; j++)
                    v = fma(left ? A.ops.DL[i][j] : A.ops.DR[i][j], f[j], v);
                double *q = acc + (i0 + i * stride) * kWarp;
                *q = d == 0 ? cd * v : fma(cd, v, *q);
            }
        }
    }
    // out = an f^n + b (f_s (1 - dt / tau) + dt (R + g / tau)), conservative Maxwellian g of the point
    int col[3];
    columns64(A.tab, slot, col);
    const double gm = A.gmask[slot], bdt = A.b * A.dt;
    const int nt = A.tab.n[0] + A.tab.n[1] + A.tab.n[2];
    double *dst = A.dst + fidx(vl, e, 0, lane, E, NP);
    double xi[3] = {0.0, 0.0, 0.0}, xs = 0.0;
    if (A.fpar)
        for (int d = 0; d < 3; d++) {
            xi[d] = A.xi[d * A.nslots + slot];
            xs = fma(xi[d], xi[d], xs);
        }
#pragma unroll 4
    for (int i = 0; i < NP; i++) {
        const int64_t pt = (int64_t)e * NP + i;
        const double *t = A.etab + ((int64_t)el * NP + i) * nt;
        const double kg = bdt * (A.itau ? A.itau[pt] : A.inv_tau);
        double w = kg * gm;
        if (A.fpar) {  // body-force source g (q0 + q . xi + q4 |xi|^2)
            const double *q = A.fpar + pt * 5;
            w = fma(bdt * gm, q[0] + q[1] * xi[0] + q[2] * xi[1] + q[3] * xi[2] + q[4] * xs, w);
        }
        double out = fma(A.b - kg, fs[i * kWarp], acc[i * kWarp]);
        out = fma(w, t[col[0]] * t[col[1]] * t[col[2]], out);
        if (fn)
            out = fma(A.an, fn[i * kWarp], out);
        dst[i * kWarp] = out;
    }
}

// The stage on curvilinear hexahedra: thread per degree of freedom.
__global__ void __launch_bounds__(256) k64_stage_curved(const Stage64Args A)
{
    const int NP = A.NP, N1 = A.N1, E = A.mesh.nelem, nt = A.tab.n[0] + A.tab.n[1] + A.tab.n[2];
    const int64_t n = (int64_t)A.nvt * A.ecount * NP * kWarp;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const int lane = (int)(q % kWarp);
        const int i = (int)((q / kWarp) % NP);
        const int el = (int)((q / ((int64_t)kWarp * NP)) % A.ecount), e = A.e0 + el;
        const int vl = (int)(q / ((int64_t)kWarp * NP * A.ecount));
        const int64_t at = fidx(vl, e, i, lane, E, NP);
        const int slot = (A.vt0 + vl) * kWarp + lane;
        const int ec[3] = {e % A.mesh.ne[0], (e / A.mesh.ne[0]) % A.mesh.ne[1], e / (A.mesh.ne[0] * A.mesh.ne[1])};
        const int ic[3] = {i % N1, (i / N1) % N1, i / (N1 * N1)};
        const double fs = A.src[at];
        double xi[3];
        for (int d = 0; d < 3; d++)
            xi[d] = A.xi[d * A.nslots + slot];
        // the reference-space flux (Ja^d . xi) f over J
        const double R = curved_residual64(A, vl, e, i, lane, slot, ec, ic, xi);
        // conservative Maxwellian of this point, BGK relaxation and the Shu-Osher combination
        int col[3];
        columns64(A.tab, slot, col);
        const double *t = A.etab + ((int64_t)el * NP + i) * nt;
        const double g = A.gmask[slot] * (t[col[0]] * t[col[1]] * t[col[2]]);
        double src = (g - fs) * (A.itau ? A.itau[(int64_t)e * NP + i] : A.inv_tau);
        if (A.fpar) {  // body-force source g (q0 + q . xi + q4 |xi|^2)
            const double *p = A.fpar + ((int64_t)e * NP + i) * 5;
            src += g * (p[0] + p[1] * xi[0] + p[2] * xi[1] + p[3] * xi[2] + p[4] * (xi[0] * xi[0] + xi[1] * xi[1] + xi[2] * xi[2]));
        }
        double out = A.b * (fs + A.dt * (R + src));
        if (A.fn)
            out += A.an * A.fn[at];
        A.dst[at] = out;
    }
}

__global__ void __launch_bounds__(256) k64_moments(const Moments64Args A)
{
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= A.npts)
        return;
    const int e = warp / A.NP, i = warp % A.NP;
    double m[5] = {0, 0, 0, 0, 0};
    for (int c = 0; c < A.nchunks; c++)
        for (int vl = 0; vl < A.nvt[c]; vl++) {
            const double v = A.base[c][fidx(vl, e, i, lane, A.E, A.NP)];
            const double *w = A.wpsi + ((int64_t)(A.vt0[c] + vl) * kWarp + lane) * 5;
            for (int q = 0; q < 5; q++)
                m[q] += w[q] * v;
        }
    for (int q = 0; q < 5; q++) {
        double v = m[q];
        for (int o = 16; o > 0; o >>= 1)
            v += __shfl_xor_sync(0xffffffffu, v, o);
        m[q] = v;
    }
    if (lane < 5)
        A.Q[(int64_t)warp * 5 + lane] = m[lane];
}

// The initial state as Maxwellian parameters par = (C, U, 1 / (2 theta)), C = rho (2 pi theta)^(-m/2).
__global__ void k64_init_par(double *par, const double *prim, int npts, int vdim, int *err)
{
    const int pt = blockIdx.x * blockDim.x + threadIdx.x;
    if (pt >= npts)
        return;
    const double *s = prim + (int64_t)pt * 5;
    double *p = par + (int64_t)pt * 5;
    const bool ok = s[0] > 0.0 && s[4] > 0.0;
    if (!ok)
        atomicOr(err, kErrDomain);
    p[0] = ok ? s[0] * pow(2.0 * 3.14159265358979323846 * s[4], -0.5 * vdim) : 0.0;
    for (int d = 0; d < 3; d++)
        p[1 + d] = ok && d < vdim ? s[1 + d] : 0.0;  // m = 2: u_z and U_z take no part
    p[4] = ok ? 0.5 / s[4] : 0.0;
}

// Sample the tabulated Maxwellians of points p0 .. p0 + np - 1 into the FP64 layout (3 operations per degree of
// freedom where an exponential and a power each took some 30).
__global__ void __launch_bounds__(256) k64_init(double *f, const double *etab, const Table64Args T, const float *gmask,
                                                int nvt, int npts, int p0, int np)
{
    const int64_t n = (int64_t)nvt * np;
    const int nt = T.n[0] + T.n[1] + T.n[2], lane = threadIdx.x & 31;
    for (int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; q < n; q += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int slot = (int)(q / np) * kWarp + lane;
        int col[3];
        columns64(T, slot, col);
        const double *t = etab + (q % np) * nt;
        f[((q / np) * npts + p0 + q % np) * kWarp + lane] = gmask[slot] * (t[col[0]] * t[col[1]] * t[col[2]]);
    }
}

// f (device tiles, FP64) <-> host-order staging [pt - p0][k] (FP64)
__global__ void k64_convert(double *f, double *st, const int *slotk, int nvt, int E, int NP, int64_t nvel, int p0,
                            int npt, int to_device)
{
    const int64_t n = (int64_t)nvt * npt * kWarp;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const int lane = (int)(q % kWarp);
        const int pl = (int)((q / kWarp) % npt);
        const int vt = (int)(q / ((int64_t)kWarp * npt));
        const int k = slotk[vt * kWarp + lane];
        const int pt = p0 + pl;
        double &v = f[fidx(vt, pt / NP, pt % NP, lane, E, NP)];
        if (to_device)
            v = k < 0 ? 0.0 : st[(int64_t)pl * nvel + k];
        else if (k >= 0)
            st[(int64_t)pl * nvel + k] = v;
    }
}

static int grid_for(int64_t n, int threads) { return (int)std::min<int64_t>((n + threads - 1) / threads, 152 * 32); }

// Zhang-Shu positivity limiter on the FP64 stage output (Sec. 2.1, Eqs. 10-11): thread per
// (tile, element, lane); the element mean uses the Gauss-Legendre weights of the nodes.
__global__ void __launch_bounds__(256) k64_limit(double *f, int nvt, int E, int NP, int N1, int dim, Ops64 ops,
                                                 const double *ijac)
{
    const int64_t n = (int64_t)nvt * E * kWarp;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const int lane = (int)(q % kWarp);
        const int64_t ve = q / kWarp;  // (tile, element)
        double *b = f + ve * NP * kWarp + lane;
        double mean = 0.0, wsum = 0.0, mn = b[0];
        for (int i = 0; i < NP; i++) {
            double w = ops.wq[i % N1];
            if (dim >= 2)
                w *= ops.wq[(i / N1) % N1];
            if (dim >= 3)
                w *= ops.wq[i / (N1 * N1)];
            if (ijac)  // curvilinear: the physical element's mean (weights W J)
                w /= ijac[(ve % E) * NP + i];
            const double v = b[(int64_t)i * kWarp];
            mean += w * v;
            wsum += w;
            mn = fmin(mn, v);
        }
        mean /= wsum;
        if (!(mn < 0.0))
            continue;
        const double beta = fmin(fabs(mean / (mean - mn)), 1.0);
        for (int i = 0; i < NP; i++)
            b[(int64_t)i * kWarp] = mean + beta * (b[(int64_t)i * kWarp] - mean);
    }
}

cudaError_t launch_limit64(double *f, int nvt, int E, int NP, int N1, int dim, const Ops64 &ops, const double *ijac,
                           cudaStream_t s)
{
    const int64_t n = (int64_t)nvt * E * kWarp;
    const int blocks = (int)std::min<int64_t>((n + 255) / 256, 152 * 16);
    k64_limit<<<blocks, 256, 0, s>>>(f, nvt, E, NP, N1, dim, ops, ijac);
    return cudaGetLastError();
}

template <int N1>
static cudaError_t stage64(const Stage64Args &A, cudaStream_t s)
{
    const int smem = A.NP * kWarp * (int)sizeof(double);  // at most 16 KB (p = 3, 3-D)
    k64_stage<N1><<<A.nvt * A.ecount, kWarp, smem, s>>>(A);
    return cudaGetLastError();
}

cudaError_t launch_stage64(const Stage64Args &A, cudaStream_t s)
{
    if (A.ja) {
        k64_stage_curved<<<grid_for((int64_t)A.nvt * A.ecount * A.NP * kWarp, 256), 256, 0, s>>>(A);
        return cudaGetLastError();
    }
    switch (A.N1) {
    case 2: return stage64<2>(A, s);
    case 3: return stage64<3>(A, s);
    case 4: return stage64<4>(A, s);
    case 5: return stage64<5>(A, s);
    default: return stage64<6>(A, s);
    }
}

cudaError_t launch_table64(double *tab, const double *par, const Table64Args &T, int npts, cudaStream_t s)
{
    k64_table<<<grid_for((int64_t)npts * (T.n[0] + T.n[1] + T.n[2]), 256), 256, 0, s>>>(tab, par, T, npts);
    return cudaGetLastError();
}

cudaError_t launch_moments64(const Moments64Args &A, cudaStream_t s)
{
    k64_moments<<<(int)(((int64_t)A.npts * kWarp + 255) / 256), 256, 0, s>>>(A);
    return cudaGetLastError();
}

// f sampled from prim by blocks of at most `block` points, which tab holds: par and tab (the next solve's parameters and
// tables) take the intermediate values.
cudaError_t launch_init64(double *f, const double *prim, double *par, double *tab, const Table64Args &T,
                          const float *gmask, int nvt, int npts, int block, int vdim, int *err, cudaStream_t s)
{
    k64_init_par<<<(npts + 127) / 128, 128, 0, s>>>(par, prim, npts, vdim, err);
    cudaError_t e = cudaGetLastError();
    for (int64_t p0 = 0; p0 < npts && e == cudaSuccess; p0 += block) {
        const int np = (int)std::min<int64_t>(block, npts - p0);
        e = launch_table64(tab, par + p0 * 5, T, np, s);
        if (e != cudaSuccess)
            break;
        k64_init<<<grid_for((int64_t)nvt * np * kWarp, 256), 256, 0, s>>>(f, tab, T, gmask, nvt, npts, (int)p0, np);
        e = cudaGetLastError();
    }
    return e;
}

cudaError_t launch_convert64(bool to_device, double *f, double *st, const int *slotk, int nvt, int E, int NP,
                             int64_t nvel, int p0, int npt, cudaStream_t s)
{
    const int64_t n = (int64_t)nvt * npt * kWarp;
    k64_convert<<<grid_for(n, 256), 256, 0, s>>>(f, st, slotk, nvt, E, NP, nvel, p0, npt, to_device ? 1 : 0);
    return cudaGetLastError();
}

}  // namespace bgk
