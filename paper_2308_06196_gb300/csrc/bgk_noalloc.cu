// bgk_noalloc.cu -- bgk_equilibrium_noalloc: the moments + conservative-Maxwellian pass for callers
// that cannot allocate device memory.
//
// Why: some callers cannot call cudaMalloc at all -- for example code that runs inside another
// framework's memory pool or allocator hooks, under a strict no-allocation policy after start-up,
// or in a process that must not grow its device footprint after it has been sized. The regular
// path (bgk_create) allocates its own buffers, so those callers could not use it. This entry point
// allocates nothing: the caller passes device pointers for the input and the outputs, and the only
// scratch (the partial moment sums and the solver's private per-point table) lives in one
// file-scope __device__ array of fixed size. A device holds it from the moment this library's module
// is loaded there until the process exits; under lazy module loading (the CUDA default since 12.2)
// that is the first call of this entry point on the device, which is therefore the sizing point: a
// caller with a fixed footprint makes it during start-up. The call is synchronous (it reads the
// status word back), so it cannot be captured in a CUDA graph; on a capturing stream it returns
// BGK_EINVAL before enqueuing anything.
//
// Scratch layout (floats): [0, 64) status word, then partial sums [ngroups][5][npts], then the
// per-point exponent table [npts][8] written by the Newton kernel.
#include <algorithm>
#include <cstdio>
#include <mutex>

#include "bgk.h"
#include "bgk_common.cuh"

namespace bgk {
cudaError_t launch_newton(const NewtonArgs &A, cudaStream_t s);
}
using namespace bgk;

namespace {

constexpr int64_t kScratchFloats = BGK_NOALLOC_SCRATCH_BYTES / 4;
constexpr int kGroupVel = 2048;   // velocities per partial-sum group
constexpr int kStatusFloats = 64; // status word region (keeps the partials 256-byte aligned)

static __device__ __align__(256) float g_scratch[kScratchFloats];

// Per-device address of g_scratch. Host code must not use the symbol itself: on the host it names
// a stand-in object, not device memory.
std::mutex g_mu;
float *g_ptr[256] = {nullptr};

constexpr int kPartThreads = 256;               // 8 warps
constexpr int kVpt = kGroupVel / kPartThreads;  // velocities per thread: 8
constexpr int kPtBatch = 6;                     // points whose 30 sums one warp reduces together

// Partial grid-index moments sum_k W_k (1, m, sum_d r_d m_d^2) f[pt][k] (the basis of the Newton
// kernel's input, exact FP32 weights). f is in the host order [npts][N_v] with k = kx + nx (ky + ny kz).
// One CTA per (velocity group, run of ppc points): a thread owns the group's velocities tid + 256 j,
// whose five weights stay in registers for all of the CTA's points, so that a value costs its load and
// five FMAs and the reading of f is what is left. Six points at a time: their 30 sums are reduced over
// the warp by halving (lane l ends up with value l: 31 shuffles for 30 sums instead of 150), then over
// the 8 warps through shared memory. Every sum is formed in the order of one thread's eight velocities,
// the lane tree 16, 8, 4, 2, 1 and the warps in turn, whatever the number of points per CTA.
// Bound: HBM. 32,768 points of 24^3 velocities (1.81 GB): 2.54 ms with one CTA per point and group
// (index divisions and FP64 end factors per value: 0.71 TB/s), now 0.31 ms (5.8 TB/s).
__global__ void __launch_bounds__(kPartThreads, 2)
    k_noalloc_partials(const float *__restrict__ f, int npts, int ppc, int nx, int ny, int nz, float ry, float rz,
                       float *partial)
{
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, g = blockIdx.x;
    const int64_t nvel = (int64_t)nx * ny * nz;
    const int64_t k0 = (int64_t)g * kGroupVel + tid;
    float wt[kVpt][5];
    bool in[kVpt];
#pragma unroll
    for (int j = 0; j < kVpt; j++) {
        const int64_t k = k0 + j * kPartThreads;
        in[j] = k < nvel;
        const int kx = (int)(k % nx), ky = (int)((k / nx) % ny), kz = (int)(k / ((int64_t)nx * ny));
        const float W = (float)(end_factor(kx, nx) * end_factor(ky, ny) * end_factor(kz, nz));
        const float mx = (float)(2 * kx - (nx - 1)), my = (float)(2 * ky - (ny - 1)), mz = (float)(2 * kz - (nz - 1));
        wt[j][0] = W;
        wt[j][1] = W * mx;
        wt[j][2] = W * my;
        wt[j][3] = W * mz;
        wt[j][4] = W * (mx * mx + ry * (my * my) + rz * (mz * mz));
    }
    __shared__ float red[2][kPartThreads / kWarp][kWarp];
    const int p0 = blockIdx.y * ppc, p1 = min(p0 + ppc, npts);
    int buf = 0;
    for (int pb = p0; pb < p1; pb += kPtBatch, buf ^= 1) {
        float v[kPtBatch][kVpt];
#pragma unroll
        for (int q = 0; q < kPtBatch; q++) {
            const float *src = f + (int64_t)min(pb + q, p1 - 1) * nvel;
#pragma unroll
            for (int j = 0; j < kVpt; j++)  // past the last velocity: 0 (finite weights, no contribution)
                v[q][j] = in[j] ? __ldcs(src + k0 + j * kPartThreads) : 0.f;
        }
        float r[kWarp];  // value 5 q + c: moment c of point pb + q
        r[30] = r[31] = 0.f;
#pragma unroll
        for (int q = 0; q < kPtBatch; q++)
#pragma unroll
            for (int c = 0; c < 5; c++) {
                float s = 0.f;
#pragma unroll
                for (int j = 0; j < kVpt; j++)
                    s = fmaf(wt[j][c], v[q][j], s);
                r[5 * q + c] = s;
            }
        // halving reduction: after the step of distance o a lane keeps the o values whose index agrees
        // with its own bits, so lane l ends with the sum of value l
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int i = 0; i < o; i++) {
                const float keep = up ? r[i + o] : r[i], give = up ? r[i] : r[i + o];
                r[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
        }
        red[buf][w][lane] = r[0];
        __syncthreads();  // the other buffer's readers are past the barrier of the previous batch
        if (tid < 30 && pb + tid / 5 < p1) {
            float s = 0.f;
#pragma unroll
            for (int q = 0; q < kPartThreads / kWarp; q++)
                s += red[buf][q][tid];
            partial[((int64_t)g * 5 + tid % 5) * npts + pb + tid / 5] = s;
        }
    }
}

}  // namespace

extern "C" int bgk_equilibrium_noalloc(const float *d_f, int64_t npts, const bgk_vgrid *vg, double *d_Q,
                                       double *d_prim, void *stream)
{
    if (!d_f || !vg || !d_Q || !d_prim || npts < 1 || npts > (1 << 30))
        return BGK_EINVAL;
    const int vdim = vg->n[2] == 1 ? 2 : 3;  // n[2] = 1: the two-dimensional velocity space
    bool all_two = true;  // two nodes on every axis: the energy moment depends on the others
    for (int d = 0; d < vdim; d++) {
        if (vg->n[d] < 2 || vg->n[d] > 4096 || !(vg->hi[d] > vg->lo[d]))
            return BGK_EINVAL;
        all_two = all_two && vg->n[d] == 2;
    }
    if (all_two)
        return BGK_EINVAL;
    const int64_t nvel = (int64_t)vg->n[0] * vg->n[1] * vg->n[2];
    const int64_t ng64 = (nvel + kGroupVel - 1) / kGroupVel;
    if (ng64 > 65535) {
        fprintf(stderr, "bgk_equilibrium_noalloc: %lld velocities exceed the 65535 x %d velocity limit\n",
                (long long)nvel, kGroupVel);
        return BGK_EINVAL;
    }
    const int ngroups = (int)ng64;
    const int64_t need = kStatusFloats + npts * (5 * (int64_t)ngroups + kParamStride);
    if (need > kScratchFloats) {
        fprintf(stderr,
                "bgk_equilibrium_noalloc: %lld points x %lld velocities need %lld scratch bytes, more than the "
                "fixed %lld-byte scratch (max points for this grid: %lld)\n",
                (long long)npts, (long long)nvel, (long long)(need * 4), (long long)BGK_NOALLOC_SCRATCH_BYTES,
                (long long)((kScratchFloats - kStatusFloats) / (5 * (int64_t)ngroups + kParamStride)));
        return BGK_EINVAL;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256)
        return BGK_ECUDA;
    float *scr = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        if (!g_ptr[dev]) {
            // once per device, with that device current
            float *p = nullptr;
            if (cudaGetSymbolAddress((void **)&p, g_scratch) != cudaSuccess || !p)
                return BGK_ECUDA;
            g_ptr[dev] = p;
        }
        scr = g_ptr[dev];
    }
    cudaStream_t s = (cudaStream_t)stream;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess)
        return BGK_ECUDA;
    if (cap != cudaStreamCaptureStatusNone) {
        fprintf(stderr, "bgk_equilibrium_noalloc: the call is synchronous and cannot be captured in a CUDA graph\n");
        return BGK_EINVAL;
    }
    int *status = reinterpret_cast<int *>(scr);
    float *partial = scr + kStatusFloats;
    float *param = partial + (int64_t)ngroups * 5 * npts;
    if (cudaMemsetAsync(status, 0, sizeof(int), s) != cudaSuccess)
        return BGK_ECUDA;
    double v0[3], dv[3];
    for (int d = 0; d < vdim; d++) {
        v0[d] = vg->lo[d];
        dv[d] = (vg->hi[d] - vg->lo[d]) / (vg->n[d] - 1);
    }
    if (vdim == 2) {  // one node at 0 of unit weight; dv[2] a placeholder equal to dv[0]
        v0[2] = 0.0;
        dv[2] = dv[0];
    }
    // points per CTA: enough CTAs for the chip (eight per SM), whole batches of points, so that a thread's
    // weights serve many points; grid.y stays within its limit of 65535
    const int64_t per = npts * ngroups / (152 * 8) + 1;
    int64_t ppc = std::max<int64_t>(per, (npts + 65534) / 65535);
    ppc = (ppc + kPtBatch - 1) / kPtBatch * kPtBatch;
    const dim3 grid((unsigned)ngroups, (unsigned)((npts + ppc - 1) / ppc));
    const float ry = index_r(dv[1], dv[0]), rz = index_r(dv[2], dv[0]);
    k_noalloc_partials<<<grid, kPartThreads, 0, s>>>(d_f, (int)npts, (int)ppc, vg->n[0], vg->n[1], vg->n[2], ry, rz,
                                                     partial);
    if (cudaGetLastError() != cudaSuccess)
        return BGK_ECUDA;
    NewtonArgs N{};
    N.partial = partial;
    N.ngroups = ngroups;
    N.npts = (int)npts;
    N.Q = d_Q;
    N.prim = d_prim;
    N.param = param;
    N.err = status;
    N.cold = 1;
    N.it32 = 2;
    N.it64 = 1;
    for (int d = 0; d < 3; d++)
        newton_axis(N, d, v0[d], dv[d], vg->n[d]);
    N.vdim = vdim;
    if (launch_newton(N, s) != cudaSuccess)
        return BGK_ECUDA;
    int h = 0;
    if (cudaMemcpyAsync(&h, status, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return BGK_ECUDA;
    if (h & kErrDomain)
        return BGK_EDOMAIN;
    if (h & kErrNewton)
        return BGK_ENEWTON;
    return BGK_OK;
}
