// k_stage3c.cuh -- the fused SSP-RK3 stage kernel of curvilinear hexahedra on the structured element
// grid (FP32-split form), every operand staged in shared memory by bulk asynchronous copies; instantiated
// per degree in k_stage3_p*.cu.
#pragma once
#include <type_traits>

#include "k_stage3s.cuh"

#ifndef BGK_STAGE3C_MINCTAS_P3
#define BGK_STAGE3C_MINCTAS_P3 4
#endif

namespace bgk {

// ------------------------------------------------------------------------------------------------
// Curvilinear hexahedra, structured element grid (Sec. 2.1, Eqs. 6-9 on the mapped element): the
// reference-space flux u f with u = Ja^d . xi at every node, and the upwind common flux of every face
// point from the sign of the shared face normal's N . xi per lane. Layout and
// copy schedule: one CTA per (element, run of G velocity tiles), one warp per z-layer, lane = velocity of
// the tile; the warp's f_s layer double-buffered, three rotating slots per warp for f^n and the upwind
// neighbours' layers, the velocity tables double-buffered by warp 0. The staged neighbour of direction
// d is the one on the side the tile's sign octant makes upwind (the low side where xi_d >= 0): a face
// normal of a curved element is close to its axis, so that side's face is the inflow face of nearly
// every lane. A lane whose flow enters through the other face (a normal tilted against a small xi_d)
// reads that neighbour's trace from global memory; where no lane of the warp does, nothing is read.
// ------------------------------------------------------------------------------------------------
template <int N1, int GEN>
struct Stage3cSmem {
    static constexpr int NP = N1 * N1 * N1, NQ = N1 * N1;
    float fs[2][NP][kWarp];
    float sl[N1][3][NQ][kWarp];
    float tab[2][kTabRows][kWarp];
    float par[N1][(NQ + 1) / 2][kParamStride][2];  // BGK exponents by layer and node pair
    float fpar[GEN ? NP : 1][GEN ? kParamStride : 4];
    float lim[GEN ? 2 : 1][GEN ? N1 : 1][GEN ? kWarp : 4];
    float4 met[NP][3];      // metric rows Ja^d; .w of row 0 = -b dt / J (the line sums' factor), of row 1 = W J
    // where N1 is even, the rows of direction d again by the node pairs of two adjacent lines (see
    // pair_row): (x_a, x_b, y_a, y_b), (z_a, z_b, s_a, s_b) with s = -b dt / J
    float4 metp[N1 % 2 == 0 ? 3 : 1][N1 % 2 == 0 ? NP / 2 : 1][2];
    float4 fnm[3][2][NQ];   // shared face normals (direction, low/high side, face point)
    // where N1 is even, again by face-point pairs (fp, fp + 1) of the paired lines: (x_a, x_b, y_a, y_b),
    // (z_a, z_b, 0, 0)
    float4 fnmp[N1 % 2 == 0 ? 3 : 1][2][N1 % 2 == 0 ? NQ / 2 : 1][2];
    float iwj;              // 1 / sum_i W_i J_i
    unsigned long long bar[N1][5];
    unsigned long long tbar[2];
};

// The reference-space line of direction d at one lane: node values fl, fluxes u fl, the exterior
// traces tL / tR used where the face normal's flow enters (uL > 0 at the low face, uR < 0 at the high
// face), the element's own trace of f elsewhere (as curv_line in k_stage3.cuh).
template <int N1>
__device__ __forceinline__ void curv_line_c(float (&sv)[N1], const float (&fl)[N1], const float (&u)[N1], float uL,
                                            float uR, float tL, float tR, const Ops &op)
{
    float F[N1], oL = 0.f, oR = 0.f;
#pragma unroll
    for (int j = 0; j < N1; j++) {
        F[j] = u[j] * fl[j];
        oL = fmaf(op.lm[j], fl[j], oL);
        oR = fmaf(op.lp[j], fl[j], oR);
    }
    const float FIL = uL * (uL > 0.f ? tL : oL);
    const float FIR = uR * (uR < 0.f ? tR : oR);
#pragma unroll
    for (int i = 0; i < N1; i++) {
        float a = fmaf(op.gl[i], FIL, op.gr[i] * FIR);
#pragma unroll
        for (int j = 0; j < N1; j++)
            a = fmaf(op.DM[i][j], F[j], a);
        sv[i] = a;
    }
}

// Node pairs of the paired lines of direction d (N1 even): lines 2 lp and 2 lp + 1 of a warp, node j:
// the pair's first node a (its partner a + N1 for d = 0, a + 1 otherwise) and its slot in metp[d].
template <int N1>
__host__ __device__ constexpr int pair_row(int d, int a)
{
    return d == 0 ? a % N1 + N1 * ((a / N1) % N1 / 2) + (N1 * N1 / 2) * (a / (N1 * N1))
                  : (a % N1) / 2 + (N1 / 2) * (a / N1);
}

// GEN = 0: every face periodic, no body force, no limiter, constant tau and one velocity spacing on all
// axes (the lean form of k_stage3s); GEN = 1: Dirichlet and diffuse-wall ghosts, the force source, the
// limiter, variable tau and per-axis spacings.
template <int N1, int GEN>
__global__ void __launch_bounds__(kWarp *N1, (N1 >= 4 ? BGK_STAGE3C_MINCTAS_P3 : (N1 == 3 ? 6 : 8))) k_stage3c(const StageArgs A)
{
    constexpr int NQ = N1 * N1;
    constexpr int NP = NQ * N1;
    constexpr int NT = kWarp * N1;
    constexpr uint32_t kRow = kWarp * sizeof(float);
    using Sm = Stage3cSmem<N1, GEN>;
    extern __shared__ __align__(16) unsigned char smraw[];
    Sm &sm = *reinterpret_cast<Sm *>(smraw);

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int E = A.mesh.nelem;
    const int gl = blockIdx.x / E;
    const int e = blockIdx.x % E;
    int vl0, vl1;
    task_tiles(A, gl, vl0, vl1);
    int ge = min(vl0 + A.G, vl1);  // end of the moment group
    int ec[3];
    ec[0] = e % A.mesh.ne[0];
    ec[1] = (e / A.mesh.ne[0]) % A.mesh.ne[1];
    ec[2] = e / (A.mesh.ne[0] * A.mesh.ne[1]);
    const float bdt = A.b * A.dt;

    // the element's BGK exponents, body-force polynomials, metric rows and face normals
    {
        constexpr int NH = (NQ + 1) / 2;
        const float *src = A.param + (int64_t)e * NP * kParamStride;
        for (int q = tid; q < N1 * NH * 2 * kParamStride; q += NT) {
            const int c = q % kParamStride, sl = (q / kParamStride) & 1, h = (q / (2 * kParamStride)) % NH;
            const int lw = q / (2 * kParamStride * NH);
            const int node = lw * NQ + min(2 * h + sl, NQ - 1);
            sm.par[lw][h][c][sl] = __ldg(src + node * kParamStride + c);
        }
        if (GEN && A.fpar) {
            const float4 *f4 = reinterpret_cast<const float4 *>(A.fpar + (int64_t)e * NP * kParamStride);
            float4 *d4 = reinterpret_cast<float4 *>(&sm.fpar[0][0]);
            for (int q = tid; q < NP * kParamStride / 4; q += NT)
                d4[q] = __ldg(f4 + q);
        }
        for (int q = tid; q < NP * 3; q += NT) {
            float4 m = __ldg(A.met + (int64_t)e * NP * 3 + q);
            if (q % 3 == 0)
                m.w = -bdt * m.w;  // rounded as the product the unstaged kernel forms at every use
            (&sm.met[0][0])[q] = m;
        }
        if constexpr (N1 % 2 == 0) {
            for (int q = tid; q < 3 * NP; q += NT) {  // q = d NP + node a; the pair's first nodes only
                const int d = q / NP, a = q % NP;
                const bool first = d == 0 ? ((a / N1) % N1) % 2 == 0 : (a % N1) % 2 == 0;
                if (!first)
                    continue;
                const int bn = a + (d == 0 ? N1 : 1);
                const float4 ma = __ldg(A.met + ((int64_t)e * NP + a) * 3 + d);
                const float4 mb = __ldg(A.met + ((int64_t)e * NP + bn) * 3 + d);
                const float sa = -bdt * __ldg(A.met + ((int64_t)e * NP + a) * 3).w;
                const float sb = -bdt * __ldg(A.met + ((int64_t)e * NP + bn) * 3).w;
                sm.metp[d][pair_row<N1>(d, a)][0] = make_float4(ma.x, mb.x, ma.y, mb.y);
                sm.metp[d][pair_row<N1>(d, a)][1] = make_float4(ma.z, mb.z, sa, sb);
            }
        }
        for (int q = tid; q < 6 * NQ; q += NT)
            (&sm.fnm[0][0][0])[q] = __ldg(A.fnm + (int64_t)e * 6 * NQ + q);
        if constexpr (N1 % 2 == 0) {
            for (int q = tid; q < 3 * NQ; q += NT) {  // q = (d, side) NQ / 2 + pair
                const int ds = q / (NQ / 2), pr = q % (NQ / 2);
                const float4 na = __ldg(A.fnm + (int64_t)e * 6 * NQ + ds * NQ + 2 * pr);
                const float4 nb = __ldg(A.fnm + (int64_t)e * 6 * NQ + ds * NQ + 2 * pr + 1);
                sm.fnmp[ds / 2][ds % 2][pr][0] = make_float4(na.x, nb.x, na.y, nb.y);
                sm.fnmp[ds / 2][ds % 2][pr][1] = make_float4(na.z, nb.z, 0.f, 0.f);
            }
        }
        if (tid == 0)
            sm.iwj = __ldg(A.iwj + e);
    }
    const uint32_t bar0 = smem_u32(&sm.bar[w][0]), tbar0 = smem_u32(&sm.tbar[0]);
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    auto tbar = [&](int b) { return tbar0 + 8u * (uint32_t)b; };
    if (lane == 0) {
#pragma unroll
        for (int i = 0; i < 5; i++)
            mbar_init(bar(i), 1);
        if (w == 0) {
            mbar_init(tbar(0), 1);
            mbar_init(tbar(1), 1);
        }
        fence_mbar_init();
    }
    __syncthreads();

    const bool has_fn = A.fn != nullptr;
    // the staged (octant-upwind) neighbour of every direction of tile vl, -1 on a Dirichlet or wall face
    auto nbrs_oct = [&](int oct, int (&en)[3]) {
#pragma unroll
        for (int d = 0; d < 3; d++)
            en[d] = upwind_neighbour(A.mesh, ec, d, ((oct >> d) & 1) != 0);
    };
    auto nbrs = [&](int vl, int (&en)[3]) {
        const int oct = (int)__ldg(A.toct + A.vt0 + vl);
#pragma unroll
        for (int d = 0; d < 3; d++)
            en[d] = upwind_neighbour(A.mesh, ec, d, ((oct >> d) & 1) != 0);
    };
    // role lanes: lane 0 the f_s layer, RZ .. RZ + N1 - 1 the z-neighbour's row groups,
    // RFN the f^n layer, RX / RY the x- / y-neighbour's layer w, RT of warp 0 the velocity table
    constexpr int RZ = 1, RFN = N1 + 1, RX = N1 + 2, RY = N1 + 3, RT = N1 + 4;
    const int64_t tstride = (int64_t)E * NP * kWarp;
    auto role_src = [&](const int (&en)[3]) -> const float * {
        if (lane == 0)
            return A.src + fidx(0, e, NQ * w, 0, E, NP);
        if (lane >= RZ && lane < RZ + N1)
            return en[2] >= 0 ? A.src + fidx(0, en[2], N1 * w + NQ * (lane - RZ), 0, E, NP) : nullptr;
        if (lane == RFN)
            return A.fn ? A.fn + fidx(0, e, NQ * w, 0, E, NP) : nullptr;
        if (lane == RX)
            return en[0] >= 0 ? A.src + fidx(0, en[0], NQ * w, 0, E, NP) : nullptr;
        if (lane == RY)
            return en[1] >= 0 ? A.src + fidx(0, en[1], NQ * w, 0, E, NP) : nullptr;
        return nullptr;
    };
    const uint32_t fs0 = smem_u32(&sm.fs[0][NQ * w][0]), sl0 = smem_u32(&sm.sl[w][0][0][0]);
    constexpr uint32_t kFsBuf = NP * kRow, kSlot = NQ * kRow;
    auto issue_layer = [&](const float *csrc, int vl, int k) {
        const uint32_t bb = bar(2 + k);
        mbar_arrive_expect_tx(bb, csrc ? kSlot : 0);
        if (csrc)
            bulk_g2s(sl0 + k * kSlot, csrc + vl * tstride, kSlot, bb);
    };

    int en[3];
    nbrs(vl0, en);
    const float *csrc = role_src(en);
    // the neighbours and the role lanes' sources are recomputed only where the octant changes from one
    // tile to the next (the velocities are ordered by octant, so within a chunk almost never)
    int octc = (int)__ldg(A.toct + A.vt0 + vl0);
    const float *fsrc = A.src + fidx(0, e, NQ * w, 0, E, NP);  // lane 0's source (the same every tile)
    if (lane == 0) {
        mbar_arrive_expect_tx(bar(0), kSlot);
        bulk_g2s(fs0, fsrc + vl0 * tstride, kSlot, bar(0));
        if (w == 0) {
            mbar_arrive_expect_tx(tbar(0), kTabRows * kRow);
            bulk_g2s(smem_u32(&sm.tab[0][0][0]), A.vtab + (int64_t)(A.vt0 + vl0) * kTabRows * kWarp,
                     kTabRows * kRow, tbar(0));
        }
    }
    if (lane == RFN && has_fn)
        issue_layer(csrc, vl0, 0);
    if (lane == RX)
        issue_layer(csrc, vl0, 1);
    if (lane == RY)
        issue_layer(csrc, vl0, 2);
    uint32_t ph = 0;
    auto wait = [&](int i) {
        mbar_wait(bar(i), (ph >> i) & 1, A.err);
        ph ^= 1u << i;
    };

    const int np = lane >> 2, kg = lane & 3;
    constexpr int NHR = NQ > 8 ? 2 : 1;
    float msum[NHR][5];
#pragma unroll
    for (int h = 0; h < NHR; h++)
#pragma unroll
        for (int c = 0; c < 5; c++)
            msum[h][c] = 0.f;
    const float kb = A.kb;

    int ka = 0;
    for (int vl = vl0; vl < vl1;) {  // a moment group
        for (; vl < ge; vl++) {
            const int vt = A.vt0 + vl;
            const int slot = vt * kWarp + lane;
            const int b = (vl - vl0) & 1;
            const int kx = ka == 2 ? 0 : ka + 1, ky = ka == 0 ? 2 : ka - 1;
            int enn[3] = {en[0], en[1], en[2]};
            const bool more = vl + 1 < vl1;
            const int octn = more ? (int)__ldg(A.toct + vt + 1) : octc;
            const bool turn = octn != octc;  // the next tile lies in another octant
            if (turn)
                nbrs_oct(octn, enn);
            __syncwarp();
            if (lane == 0 && more) {
                fence_proxy_async();
                mbar_arrive_expect_tx(bar(b ^ 1), kSlot);
                bulk_g2s(fs0 + (b ^ 1) * kFsBuf, fsrc + (vl + 1) * tstride, kSlot, bar(b ^ 1));
            }
            const int oct = octc;
            const bool l0 = (oct & 1) != 0, l1 = (oct & 2) != 0, l2 = (oct & 4) != 0;
            const int enx = en[0], eny = en[1], enz = en[2];

            wait(b);
            mbar_wait(tbar(b), (ph >> (5 + b)) & 1, A.err);
            ph ^= 1u << (5 + b);
            const float m0 = sm.tab[b][0][lane], m1 = sm.tab[b][1][lane], m2 = sm.tab[b][2][lane];
            const float x0 = fmaf(A.vs[0], m0, A.vc[0]), x1 = fmaf(A.vs[1], m1, A.vc[1]), x2 = fmaf(A.vs[2], m2, A.vc[2]);
            float acc[NQ];
            if (has_fn) {
                wait(2 + ka);
#pragma unroll
                for (int q = 0; q < NQ; q++)
                    acc[q] = sm.sl[w][ka][q][lane];
            } else {
#pragma unroll
                for (int q = 0; q < NQ; q++)
                    acc[q] = 0.f;
            }
            // slot ka is consumed: the z-neighbour's slice lands there
            __syncwarp();
            if (lane >= RZ && lane < RZ + N1) {
                const float *zs = csrc;
                const uint32_t bb = bar(2 + ka);
                fence_proxy_async();
                if (lane == RZ)
                    mbar_arrive_expect_tx(bb, zs ? kSlot : 0);
                if (zs)
                    bulk_g2s(sl0 + ka * kSlot + (lane - RZ) * N1 * kRow, zs + vl * tstride, N1 * kRow, bb);
            }
            // (launch-uniform feature tests sit outside the unrolled node loops, which stay one basic block)
            if (GEN && A.vtau) {
#pragma unroll
                for (int q = 0; q < NQ; q++)
                    acc[q] = fmaf(A.an, acc[q],
                                  __fsub_rn(A.b, __fmul_rn(bdt, sm.par[w][q / 2][6][q % 2])) * sm.fs[b][q + NQ * w][lane]);
            } else {
#pragma unroll
                for (int q = 0; q < NQ; q++)
                    acc[q] = fmaf(A.an, acc[q], kb * sm.fs[b][q + NQ * w][lane]);
            }
            // The lines of direction d through this warp's nodes: x- and y-lines of layer w (their sums
            // go to acc), z-lines of slice w (their sums overwrite the rows they read, after B1). Line ln
            // has face point fp = ln + N1 w on both faces. lo: the tile's octant stages the low-side
            // neighbour (slot ks); es: that neighbour, < 0 on a boundary face (its ghost value instead).
            // Lanes whose flow enters through the other face take that face's exterior trace, read for all
            // lines of the direction at once and only where some lane of the warp needs it.
            auto lines = [&](auto dc, int ks, bool lo, int es) {
                constexpr int d = decltype(dc)::value;
                auto node = [&](int ln, int j) {  // element node j of line ln
                    return d == 0 ? j + N1 * ln + NQ * w : (d == 1 ? ln + N1 * j + NQ * w : ln + N1 * w + NQ * j);
                };
                auto srow = [&](int ln, int j) { return d == 0 ? j + N1 * ln : ln + N1 * j; };  // row in slot ks
                float cS[N1], cF[N1];  // trace weights of the staged and of the other side's neighbour
#pragma unroll
                for (int j = 0; j < N1; j++) {
                    cS[j] = lo ? A.ops.lp[j] : A.ops.lm[j];
                    cF[j] = lo ? A.ops.lm[j] : A.ops.lp[j];
                }
                auto trace = [&](const float(&v)[N1], const float(&c)[N1]) {  // trace_line with weights c
                    float t = 0.f;
#pragma unroll
                    for (int j = 1; j < N1; j++)
                        t = fmaf(c[j], v[j] - v[0], t);
                    return v[0] + t;
                };
                float uL[N1], uR[N1], tF[N1];
                bool far = false;
                if constexpr (N1 % 2 == 0) {  // two face points at a time (the same operations per half)
                    const unsigned long long X0 = pack2(x0, x0), X1 = pack2(x1, x1), X2 = pack2(x2, x2);
#pragma unroll
                    for (int ln = 0; ln < N1; ln += 2) {
                        const int pr = (ln + N1 * w) / 2;
                        float u2[2][2];
#pragma unroll
                        for (int sd = 0; sd < 2; sd++) {
                            const float4 n0 = sm.fnmp[d][sd][pr][0], n1 = sm.fnmp[d][sd][pr][1];
                            unpack2(ffma2(pack2(n1.x, n1.y), X2, ffma2(pack2(n0.z, n0.w), X1, fmul2(pack2(n0.x, n0.y), X0))),
                                    u2[sd][0], u2[sd][1]);
                        }
#pragma unroll
                        for (int h = 0; h < 2; h++) {
                            uL[ln + h] = u2[0][h];
                            uR[ln + h] = u2[1][h];
                            tF[ln + h] = 0.f;
                            far = far || (lo ? uR[ln + h] < 0.f : uL[ln + h] > 0.f);
                        }
                    }
                } else {
#pragma unroll
                    for (int ln = 0; ln < N1; ln++) {
                        const int fp = ln + N1 * w;
                        const float4 nL = sm.fnm[d][0][fp], nR = sm.fnm[d][1][fp];
                        uL[ln] = fmaf(nL.z, x2, fmaf(nL.y, x1, nL.x * x0));
                        uR[ln] = fmaf(nR.z, x2, fmaf(nR.y, x1, nR.x * x0));
                        tF[ln] = 0.f;
                        far = far || (lo ? uR[ln] < 0.f : uL[ln] > 0.f);
                    }
                }
                if (__any_sync(0xffffffffu, far)) {
                    const int g = 2 * d + (lo ? 1 : 0);
                    const int eo = upwind_neighbour(A.mesh, ec, d, !lo);
                    if (!GEN || eo >= 0) {
                        const float *nb = A.src + fidx(vl, eo, 0, lane, E, NP);
                        float v[N1][N1];
#pragma unroll
                        for (int ln = 0; ln < N1; ln++) {
                            const bool need = lo ? uR[ln] < 0.f : uL[ln] > 0.f;
#pragma unroll
                            for (int j = 0; j < N1; j++)
                                v[ln][j] = need ? __ldg(nb + node(ln, j) * kWarp) : 0.f;
                        }
#pragma unroll
                        for (int ln = 0; ln < N1; ln++)
                            tF[ln] = trace(v[ln], cF);
                    } else {
                        // (the wall test is outside the loops: no load is formed from a pointer that may be null)
                        const float gv = __ldg(A.ghost + (int64_t)g * A.nslots + slot);
                        if (A.mesh.bc[g] == 2) {
                            const float *rw = A.rhow + ((int64_t)g * A.nfmax + face_elem(A.mesh, ec, d)) * NQ + N1 * w;
#pragma unroll
                            for (int ln = 0; ln < N1; ln++)
                                tF[ln] = gv * __ldg(rw + ln);
                        } else {
#pragma unroll
                            for (int ln = 0; ln < N1; ln++)
                                tF[ln] = gv;
                        }
                    }
                }
                float gS[N1];  // the staged side's ghost value of every line on a boundary face
#pragma unroll
                for (int ln = 0; ln < N1; ln++)
                    gS[ln] = 0.f;
                if (GEN && es < 0) {
                    const int g = 2 * d + (lo ? 0 : 1);
                    const float gv = __ldg(A.ghost + (int64_t)g * A.nslots + slot);
                    if (A.mesh.bc[g] == 2) {
                        const float *rw = A.rhow + ((int64_t)g * A.nfmax + face_elem(A.mesh, ec, d)) * NQ + N1 * w;
#pragma unroll
                        for (int ln = 0; ln < N1; ln++)
                            gS[ln] = gv * __ldg(rw + ln);
                    } else {
#pragma unroll
                        for (int ln = 0; ln < N1; ln++)
                            gS[ln] = gv;
                    }
                }
                if constexpr (N1 % 2 == 0) {
                    // two adjacent lines at a time on packed FP32 pairs: the same operations, in the same
                    // order, as curv_line_c on each line (bit-identical results)
                    const unsigned long long X0 = pack2(x0, x0), X1 = pack2(x1, x1), X2 = pack2(x2, x2);
#pragma unroll
                    for (int ln = 0; ln < N1; ln += 2) {
                        unsigned long long fl[N1], F[N1], v[N1], sp[N1];
#pragma unroll
                        for (int j = 0; j < N1; j++) {
                            fl[j] = pack2(sm.fs[b][node(ln, j)][lane], sm.fs[b][node(ln + 1, j)][lane]);
                            v[j] = pack2(sm.sl[w][ks][srow(ln, j)][lane], sm.sl[w][ks][srow(ln + 1, j)][lane]);
                            const float4 *mp = &sm.metp[d][pair_row<N1>(d, node(ln, j))][0];
                            const float4 p0 = mp[0], p1 = mp[1];
                            const unsigned long long u =
                                ffma2(pack2(p1.x, p1.y), X2, ffma2(pack2(p0.z, p0.w), X1, fmul2(pack2(p0.x, p0.y), X0)));
                            F[j] = fmul2(u, fl[j]);
                            sp[j] = pack2(p1.z, p1.w);
                        }
                        // the staged side's trace of both lines, and their own traces
                        unsigned long long t = 0ull, oL = 0ull, oR = 0ull;
#pragma unroll
                        for (int j = 1; j < N1; j++)
                            t = ffma2(dup2(cS[j]), fsub2(v[j], v[0]), t);
                        t = fadd2(v[0], t);
#pragma unroll
                        for (int j = 0; j < N1; j++) {
                            oL = ffma2(dup2(A.ops.lm[j]), fl[j], oL);
                            oR = ffma2(dup2(A.ops.lp[j]), fl[j], oR);
                        }
                        float tS2[2], oL2[2], oR2[2], FI[2][2];
                        unpack2(t, tS2[0], tS2[1]);
                        unpack2(oL, oL2[0], oL2[1]);
                        unpack2(oR, oR2[0], oR2[1]);
#pragma unroll
                        for (int h = 0; h < 2; h++) {
                            const float tS = !GEN || es >= 0 ? tS2[h] : gS[ln + h];
                            const float tL = lo ? tS : tF[ln + h], tR = lo ? tF[ln + h] : tS;
                            FI[0][h] = uL[ln + h] * (uL[ln + h] > 0.f ? tL : oL2[h]);
                            FI[1][h] = uR[ln + h] * (uR[ln + h] < 0.f ? tR : oR2[h]);
                        }
                        const unsigned long long FIL = pack2(FI[0][0], FI[0][1]), FIR = pack2(FI[1][0], FI[1][1]);
#pragma unroll
                        for (int i = 0; i < N1; i++) {
                            unsigned long long a = ffma2(dup2(A.ops.gl[i]), FIL, fmul2(dup2(A.ops.gr[i]), FIR));
#pragma unroll
                            for (int j = 0; j < N1; j++)
                                a = ffma2(dup2(A.ops.DM[i][j]), F[j], a);
                            float sa, sb;
                            unpack2(a, sa, sb);
                            if (d < 2) {
                                float ca, cb;
                                unpack2(sp[i], ca, cb);
                                acc[node(ln, i) - NQ * w] = fmaf(ca, sa, acc[node(ln, i) - NQ * w]);
                                acc[node(ln + 1, i) - NQ * w] = fmaf(cb, sb, acc[node(ln + 1, i) - NQ * w]);
                            } else {
                                sm.fs[b][node(ln, i)][lane] = sa;
                                sm.fs[b][node(ln + 1, i)][lane] = sb;
                            }
                        }
                    }
                } else {
#pragma unroll
                    for (int ln = 0; ln < N1; ln++) {
                        float fl[N1], u[N1], sv[N1], v[N1];
#pragma unroll
                        for (int j = 0; j < N1; j++) {
                            fl[j] = sm.fs[b][node(ln, j)][lane];
                            v[j] = sm.sl[w][ks][srow(ln, j)][lane];
                            const float4 m = sm.met[node(ln, j)][d];
                            u[j] = fmaf(m.z, x2, fmaf(m.y, x1, m.x * x0));
                        }
                        const float tS = !GEN || es >= 0 ? trace(v, cS) : gS[ln];
                        curv_line_c<N1>(sv, fl, u, uL[ln], uR[ln], lo ? tS : tF[ln], lo ? tF[ln] : tS, A.ops);
#pragma unroll
                        for (int j = 0; j < N1; j++) {
                            if (d < 2)
                                acc[node(ln, j) - NQ * w] = fmaf(sm.met[node(ln, j)][0].w, sv[j], acc[node(ln, j) - NQ * w]);
                            else
                                sm.fs[b][node(ln, j)][lane] = sv[j];
                        }
                    }
                }
            };
            wait(2 + kx);
            lines(std::integral_constant<int, 0>{}, kx, l0, enx);
            wait(2 + ky);
            lines(std::integral_constant<int, 1>{}, ky, l1, eny);
            // slots kx and ky are consumed: the next tile's f^n and x-neighbour layer land there
            __syncwarp();
            if (more && ((lane == RFN && has_fn) || lane == RX)) {
                fence_proxy_async();
                issue_layer(lane == RX && turn ? role_src(enn) : csrc, vl + 1, lane == RX ? ky : kx);
            }
            __syncthreads();  // B1: every layer of the element tile has landed
            // z-lines of slice iy = w (all layers) from the shared tile
            wait(2 + ka);
            lines(std::integral_constant<int, 2>{}, ka, l2, enz);
            // slot ka is consumed: the next tile's y-neighbour layer lands there; warp 0 also brings the next
            // tile's velocity table into the other table buffer (every warp is past B1)
            __syncwarp();
            if (more && (lane == RY || (w == 0 && lane == RT))) {
                fence_proxy_async();
                if (lane == RY) {
                    issue_layer(turn ? role_src(enn) : csrc, vl + 1, ka);
                } else {
                    mbar_arrive_expect_tx(tbar(b ^ 1), kTabRows * kRow);
                    bulk_g2s(smem_u32(&sm.tab[b ^ 1][0][0]), A.vtab + (int64_t)(vt + 1) * kTabRows * kWarp,
                             kTabRows * kRow, tbar(b ^ 1));
                }
            }
            __syncthreads();  // B2: z-sums complete
#pragma unroll
            for (int q = 0; q < NQ; q++)
                acc[q] = fmaf(sm.met[q + NQ * w][0].w, sm.fs[b][q + NQ * w][lane], acc[q]);
            __syncwarp();  // the z-sums of this layer are read before its rows take the stage output
            const float gm = sm.tab[b][3][lane] != 0.f ? 1.f : 0.f;
            const float cg = A.kg * gm, cf = bdt * gm;
            const float xs = x0 * x0 + x1 * x1 + x2 * x2;
            const float mm0 = m0 * m0, mm1 = m1 * m1, mm2 = m2 * m2, mms = mm0 + mm1 + mm2;
            const bool iso = !GEN || A.viso;
            const unsigned long long M0 = pack2(m0, m0), M1 = pack2(m1, m1), M2 = pack2(m2, m2);
            const unsigned long long U0 = iso ? pack2(mms, mms) : pack2(mm0, mm0);
            const unsigned long long U1 = iso ? U0 : pack2(mm1, mm1);
            const unsigned long long U2 = iso ? 0ull : pack2(mm2, mm2);
            float *dst = A.dst + fidx(vl, e, 0, lane, E, NP);
            float lsum = 0.f, lmin = 3.4e38f;
            auto bgk_src = [&](auto vtau_c, auto force_c, auto lim_c) {
                constexpr bool VT = decltype(vtau_c)::value, FP = decltype(force_c)::value;
                constexpr bool LIM = decltype(lim_c)::value;
#pragma unroll
                for (int h = 0; h < (NQ + 1) / 2; h++) {
                    const float4 *pp = reinterpret_cast<const float4 *>(&sm.par[w][h][0][0]);
                    const float4 p01 = pp[0], p23 = pp[1], p45 = pp[2], p67 = pp[3];
                    const unsigned long long lin =
                        ffma2(pack2(p23.z, p23.w), M2,
                              ffma2(pack2(p23.x, p23.y), M1, ffma2(pack2(p01.z, p01.w), M0, pack2(p01.x, p01.y))));
                    const unsigned long long ex =
                        GEN ? ffma2(pack2(p45.x, p45.y), U0,
                                    ffma2(pack2(p45.z, p45.w), U1, ffma2(pack2(p67.x, p67.y), U2, lin)))
                            : ffma2(pack2(p45.x, p45.y), U0, ffma2(pack2(p45.z, p45.w), U0, lin));
                    float g[2];
                    exp2_fp32x2(ex, pack2(p67.z, p67.w), g[0], g[1]);
#pragma unroll
                    for (int sl = 0; sl < 2; sl++) {
                        const int q = 2 * h + sl;
                        if (q >= NQ)
                            break;
                        const int i = q + NQ * w;
                        const float a = acc[q];
                        float gc = cg;
                        if constexpr (VT) {
                            const float itau = sl == 0 ? p67.x : p67.y;
                            gc = __fsub_rn(A.b, __fsub_rn(A.b, __fmul_rn(bdt, itau))) * gm;
                        }
                        if constexpr (FP) {
                            const float4 fq = *reinterpret_cast<const float4 *>(&sm.fpar[i][0]);
                            const float qv =
                                fmaf(sm.fpar[i][4], xs, fmaf(fq.w, x2, fmaf(fq.z, x1, fmaf(fq.y, x0, fq.x))));
                            gc = fmaf(cf, qv, gc);  // on top of the node's own Maxwellian weight
                        }
                        const float o = fmaf(gc, g[sl], a);
                        if constexpr (LIM) {
                            lsum = fmaf(sm.met[i][1].w, o, lsum);
                            lmin = fminf(lmin, o);
                        } else {
                            __stcs(dst + i * kWarp, o);
                        }
                        sm.fs[b][q + NQ * w][lane ^ (4 * (q & 7))] = o;
                    }
                }
            };
            using T_ = std::true_type;
            using F_ = std::false_type;
            if constexpr (GEN) {
                if (A.limiter) {
                    if (A.fpar)
                        A.vtau ? bgk_src(T_{}, T_{}, T_{}) : bgk_src(F_{}, T_{}, T_{});
                    else
                        A.vtau ? bgk_src(T_{}, F_{}, T_{}) : bgk_src(F_{}, F_{}, T_{});
                } else {
                    if (A.fpar)
                        A.vtau ? bgk_src(T_{}, T_{}, F_{}) : bgk_src(F_{}, T_{}, F_{});
                    else
                        A.vtau ? bgk_src(T_{}, F_{}, F_{}) : bgk_src(F_{}, F_{}, F_{});
                }
            } else {
                bgk_src(F_{}, F_{}, F_{});
            }
            if (GEN && A.limiter) {
                // Zhang-Shu (Sec. 2.1, Eqs. 10-11) over the physical element: weights W J over their sum
                sm.lim[0][w][lane] = lsum;
                sm.lim[1][w][lane] = lmin;
                __syncthreads();  // B3
                float mean = 0.f, mn = sm.lim[1][0][lane];
#pragma unroll
                for (int lw = 0; lw < N1; lw++) {
                    mean += sm.lim[0][lw][lane];
                    mn = fminf(mn, sm.lim[1][lw][lane]);
                }
                mean *= sm.iwj;
                const float beta = mn < 0.f ? fminf(fabsf(mean / (mean - mn)), 1.f) : 1.f;
                if (mn < 0.f) {
#pragma unroll
                    for (int q = 0; q < NQ; q++) {
                        float &slot_o = sm.fs[b][q + NQ * w][lane ^ (4 * (q & 7))];
                        slot_o = fmaf(beta, slot_o - mean, mean);
                    }
                }
#pragma unroll
                for (int q = 0; q < NQ; q++)
                    __stcs(dst + (q + NQ * w) * kWarp, sm.fs[b][q + NQ * w][lane ^ (4 * (q & 7))]);
            }
            // moments of this layer's nodes (Eq. 2 with Eq. 12) of the stored values
            __syncwarp();
            unsigned long long pm[2][5];
#pragma unroll
            for (int h = 0; h < NHR; h++)
#pragma unroll
                for (int c = 0; c < 5; c++)
                    pm[h][c] = 0ull;
#pragma unroll
            for (int k = 0; k < 8; k += 4) {
                const int kk = 8 * kg + k;
                unsigned long long wv[5][2];
                {
                    const float4 W4 = *reinterpret_cast<const float4 *>(&sm.tab[b][3][kk]);
                    const float4 E4 = *reinterpret_cast<const float4 *>(&sm.tab[b][4][kk]);
                    wv[0][0] = pack2(W4.x, W4.y);
                    wv[0][1] = pack2(W4.z, W4.w);
                    wv[4][0] = pack2(E4.x, E4.y);
                    wv[4][1] = pack2(E4.z, E4.w);
#pragma unroll
                    for (int d = 0; d < 3; d++) {
                        const float4 M4 = *reinterpret_cast<const float4 *>(&sm.tab[b][d][kk]);
                        wv[1 + d][0] = fmul2(pack2(W4.x, W4.y), pack2(M4.x, M4.y));
                        wv[1 + d][1] = fmul2(pack2(W4.z, W4.w), pack2(M4.z, M4.w));
                    }
                }
#pragma unroll
                for (int h = 0; h < NHR; h++) {
                    const int row = min(np + 8 * h, NQ - 1);
                    const float4 v = *reinterpret_cast<const float4 *>(&sm.fs[b][row + NQ * w][kk ^ (4 * (row & 7))]);
                    const unsigned long long v01 = pack2(v.x, v.y), v23 = pack2(v.z, v.w);
#pragma unroll
                    for (int c = 0; c < 5; c++) {
                        pm[h][c] = ffma2(wv[c][0], v01, pm[h][c]);
                        pm[h][c] = ffma2(wv[c][1], v23, pm[h][c]);
                    }
                }
            }
#pragma unroll
            for (int h = 0; h < NHR; h++)
#pragma unroll
                for (int c = 0; c < 5; c++)
                    msum[h][c] += sum2(pm[h][c]);
#pragma unroll
            for (int d = 0; d < 3; d++)
                en[d] = enn[d];
            if (turn) {
                csrc = role_src(en);
                octc = octn;
            }
            ka = ka == 2 ? 0 : ka + 1;
        }
        const int grp = moment_group(A, blockIdx.x / E, vl - 1);
#pragma unroll
        for (int h = 0; h < NHR; h++) {
            const int q = np + 8 * h;
#pragma unroll
            for (int c = 0; c < 5; c++) {
                float x = msum[h][c];
                msum[h][c] = 0.f;
                x += __shfl_xor_sync(0xffffffffu, x, 1);
                x += __shfl_xor_sync(0xffffffffu, x, 2);
                if (kg == 0 && q < NQ)
                    A.partial[((int64_t)grp * 5 + c) * A.npts + (int64_t)e * NP + q + NQ * w] = x;
            }
        }
        ge = min(ge + A.G, vl1);
    }
}

// ------------------------------------------------------------------------------------------------
// The same for p = 1 on packed pairs of velocities: k_stage3s's layout (half-warp h of warp w holds layer
// 2 w + h, lane l of it velocities 2 l and 2 l + 1), four rotating buffers, moment groups and copies, with
// the reference-space lines. A shared load returns 128 bytes per cycle, broadcast or not, so a metric row, a
// face normal or an exponent that a lane reads for one velocity costs as much as its share of f; a lane with
// two velocities halves that, and one warp holds the element. 16 x 12 x 14 elements, p = 1, 24^3 velocities,
// two steps: 15.8 -> 10.8 ms. At p = 3 it runs too, but slower (2.08 -> 2.35 ms per octant launch of
// 16^3 elements, 24^3 velocities: 92 instructions per 32 degrees of freedom at 0.4 per cycle; its 41 KB of
// shared memory leave 5 CTAs, 10 warps per SM, where its 168 registers would allow 6, and its code overflows the
// instruction cache), so p = 3 stays with the lane per velocity. A form in less shared memory was not tried.
// ------------------------------------------------------------------------------------------------
constexpr bool stage3c_pairs(int N1) { return N1 == 2; }

template <int N1, int GEN>
struct Stage3cpSmem {
    static_assert(N1 % 2 == 0, "a warp holds two layers");
    static constexpr int NP = N1 * N1 * N1, NQ = N1 * N1, NW = N1 / 2;
    static constexpr int kParLayer = NQ * kParamStride + 8;  // as Stage3sSmem
    // every member is read or written in 8- or 16-byte units
    alignas(16) float buf[4][NP][kWarp];
    alignas(16) float tab[2][kTabRows][kWarp];
    alignas(16) float par[N1 * kParLayer];
    alignas(16) float4 met[3][NP];     // metric rows Ja^d
    alignas(16) float sj[NP];          // -b dt / J of the nodes
    alignas(16) float4 fnm[3][2][NQ];  // shared face normals (direction, low/high side, face point)
    alignas(16) float fpar[GEN ? NP : 1][GEN ? kParamStride : 1];
    alignas(16) float lim[GEN ? 2 : 1][GEN ? N1 : 1][GEN ? kWarp : 1];
    float wj[GEN ? NP : 1];            // W J of the nodes
    float iwj;                         // 1 / sum_i W_i J_i
    unsigned long long bar[NW][4];
    unsigned long long tbar[2];
};

template <int N1, int GEN>
__global__ void __launch_bounds__(kWarp *N1 / 2, 16) k_stage3cp(const StageArgs A)
{
    using u64 = unsigned long long;
    constexpr int NQ = N1 * N1;
    constexpr int NP = NQ * N1;
    constexpr int NW = N1 / 2;
    constexpr int NT = kWarp * NW;
    constexpr uint32_t kRow = kWarp * sizeof(float);  // one node's row of a tile: 128 bytes
    using Sm = Stage3cpSmem<N1, GEN>;
    extern __shared__ __align__(16) unsigned char smraw[];
    Sm &sm = *reinterpret_cast<Sm *>(smraw);

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int hf = lane >> 4, c2 = 2 * (lane & 15);  // half-warp, first velocity of this lane
    const int lz = 2 * w + hf;                       // this lane's z-layer (and z-line slice iy)
    const int E = A.mesh.nelem;
    const int e = blockIdx.x % E;
    int vl0, vl1;
    task_tiles(A, blockIdx.x / E, vl0, vl1);
    int ge = min(vl0 + A.G, vl1);  // end of the moment group
    int ec[3];
    ec[0] = e % A.mesh.ne[0];
    ec[1] = (e / A.mesh.ne[0]) % A.mesh.ne[1];
    ec[2] = e / (A.mesh.ne[0] * A.mesh.ne[1]);

    const float bdt = A.b * A.dt;
    // the element's BGK exponents, force polynomials, metric rows and face normals
    {
        const float4 *src = reinterpret_cast<const float4 *>(A.param + (int64_t)e * NP * kParamStride);
        constexpr int kQ4 = NQ * kParamStride / 4;  // float4s of a layer
        for (int q = tid; q < N1 * kQ4; q += NT)
            *reinterpret_cast<float4 *>(&sm.par[(q / kQ4) * Sm::kParLayer + 4 * (q % kQ4)]) = __ldg(src + q);
        if (GEN && A.fpar) {
            const float4 *f4 = reinterpret_cast<const float4 *>(A.fpar + (int64_t)e * NP * kParamStride);
            float4 *d4 = reinterpret_cast<float4 *>(&sm.fpar[0][0]);
            for (int q = tid; q < NP * kParamStride / 4; q += NT)
                d4[q] = __ldg(f4 + q);
        }
        for (int q = tid; q < NP; q += NT) {
            float4 m[3];
#pragma unroll
            for (int d = 0; d < 3; d++)
                m[d] = __ldg(A.met + ((int64_t)e * NP + q) * 3 + d);
            if (GEN)
                sm.wj[q] = m[1].w;
            sm.sj[q] = -bdt * m[0].w;
#pragma unroll
            for (int d = 0; d < 3; d++)
                sm.met[d][q] = m[d];
        }
        for (int q = tid; q < 6 * NQ; q += NT)
            (&sm.fnm[0][0][0])[q] = __ldg(A.fnm + (int64_t)e * 6 * NQ + q);
        if (GEN && tid == 0)
            sm.iwj = __ldg(A.iwj + e);
    }
    // barrier addresses: bar(i) of this warp's part of buffer i; tbar(b) the tables'
    const uint32_t bar0 = smem_u32(&sm.bar[w][0]), tbar0 = smem_u32(&sm.tbar[0]);
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    auto tbar = [&](int b) { return tbar0 + 8u * (uint32_t)b; };
    if (lane == 0) {
#pragma unroll
        for (int i = 0; i < 4; i++)
            mbar_init(bar(i), 1);
        if (w == 0) {
            mbar_init(tbar(0), 1);
            mbar_init(tbar(1), 1);
        }
        fence_mbar_init();
    }
    __syncthreads();  // exponents and barriers visible to every warp

    const bool has_fn = A.fn != nullptr;
    // the staged (octant-upwind) neighbour of every direction, -1 on a Dirichlet or wall face
    auto nbrs = [&](int oct, int (&en)[3]) {
#pragma unroll
        for (int d = 0; d < 3; d++)
            en[d] = upwind_neighbour(A.mesh, ec, d, ((oct >> d) & 1) != 0);
    };
    // Bulk copies by role lanes, as k_stage3s
    constexpr int RZ = 1, RFN = N1 + 1, RX = N1 + 2, RY = N1 + 3, RT = N1 + 4;
    const int64_t tstride = (int64_t)E * NP * kWarp;  // floats between consecutive tiles of one element
    const int lay = 2 * NQ * w;  // the warp's first row
    auto role_src = [&](const int (&en)[3]) -> const float * {
        if (lane == 0)
            return A.src + fidx(0, e, lay, 0, E, NP);
        if (lane >= RZ && lane < RZ + N1)
            return en[2] >= 0 ? A.src + fidx(0, en[2], 2 * N1 * w + NQ * (lane - RZ), 0, E, NP) : nullptr;
        if (lane == RFN)
            return A.fn ? A.fn + fidx(0, e, lay, 0, E, NP) : nullptr;
        if (lane == RX)
            return en[0] >= 0 ? A.src + fidx(0, en[0], lay, 0, E, NP) : nullptr;
        if (lane == RY)
            return en[1] >= 0 ? A.src + fidx(0, en[1], lay, 0, E, NP) : nullptr;
        return nullptr;
    };
    const uint32_t part0 = smem_u32(&sm.buf[0][lay][0]);  // this warp's part of buffer 0
    constexpr uint32_t kBuf = NP * kRow, kPart = 2 * NQ * kRow;
    // a copy into this warp's part of buffer k (two layers; nothing at a boundary), from csrc at tile vl
    auto issue = [&](const float *from, int vl, int k) {
        const uint32_t bb = bar(k);
        mbar_arrive_expect_tx(bb, from ? kPart : 0);
        if (from)
            bulk_g2s(part0 + k * kBuf, from + vl * tstride, kPart, bb);
    };

    // the neighbours and the role lanes' sources are recomputed only where the octant changes from one
    // tile to the next (the velocities are ordered by octant, so within a chunk never)
    int octc = (int)__ldg(A.toct + A.vt0 + vl0);
    int en[3];
    nbrs(octc, en);
    const float *csrc = role_src(en);  // at tile 0
    // buffers of this tile's f_s, f^n (then the z-neighbour), x- and y-neighbour
    int bF = 0, bN = 1, bX = 2, bY = 3;
    if (lane == 0 || (lane == RFN && has_fn) || lane == RX || lane == RY)
        issue(csrc, vl0, lane == 0 ? bF : (lane == RFN ? bN : (lane == RX ? bX : bY)));
    if (tid == RT) {
        mbar_arrive_expect_tx(tbar(0), kTabRows * kRow);
        bulk_g2s(smem_u32(&sm.tab[0][0][0]), A.vtab + (int64_t)(A.vt0 + vl0) * kTabRows * kWarp, kTabRows * kRow, tbar(0));
    }
    uint32_t ph = 0;  // phase parity of every barrier, bit i for bar(i), bit 4 + b for tbar(b)
    auto wait = [&](int i) {
        mbar_wait(bar(i), (ph >> i) & 1, A.err);
        ph ^= 1u << i;
    };

    // moment sums: lane = (row np + 8 r, r < NR, of the warp's 2 NQ rows, np = lane / 4) x (velocity eighth
    // kg = lane % 4), running in registers
    const int np = lane >> 2, kg = lane & 3;
    constexpr int NR = 2 * NQ / 8;
    float msum[NR][5];
#pragma unroll
    for (int r = 0; r < NR; r++)
#pragma unroll
        for (int c = 0; c < 5; c++)
            msum[r][c] = 0.f;
    auto ld2 = [](const float *p) { return *reinterpret_cast<const u64 *>(p); };
    auto st2 = [](float *p, u64 v) { *reinterpret_cast<u64 *>(p) = v; };

    for (int vl = vl0; vl < vl1; vl++) {
        const int vt = A.vt0 + vl;
        const int slot = vt * kWarp + c2;
        const int b = (vl - vl0) & 1;
        float(*const F)[kWarp] = sm.buf[bF];  // f_s, then the z-sums, then the output
        const float(*const pN)[kWarp] = sm.buf[bN] + lay, (*const pX)[kWarp] = sm.buf[bX] + lay + hf * NQ,
                         (*const pY)[kWarp] = sm.buf[bY] + lay + hf * NQ;
        int enn[3] = {en[0], en[1], en[2]};  // the next tile's neighbours
        const bool more = vl + 1 < vl1;
        const int oct = octc, octn = more ? (int)__ldg(A.toct + vt + 1) : octc;
        const bool turn = octn != octc;
        if (turn)
            nbrs(octn, enn);

        wait(bF);
        mbar_wait(tbar(b), (ph >> (4 + b)) & 1, A.err);
        ph ^= 1u << (4 + b);
        // the two velocities: grid indices, velocities
        float m[3][2], x[3][2];
#pragma unroll
        for (int d = 0; d < 3; d++) {
            unpack2(ld2(&sm.tab[b][d][c2]), m[d][0], m[d][1]);
#pragma unroll
            for (int s = 0; s < 2; s++)
                x[d][s] = fmaf(A.vs[d], m[d][s], A.vc[d]);
        }
        u64 f[NQ], acc[NQ];
#pragma unroll
        for (int q = 0; q < NQ; q++)
            f[q] = ld2(&F[q + NQ * lz][c2]);
        // acc = an f^n + b (1 - dt/tau) f_s
        // (launch-uniform feature tests sit outside the unrolled node loops, which stay one basic block)
        if (GEN && A.vtau) {  // variable collision time: b (1 - dt/tau) of every node
#pragma unroll
            for (int q = 0; q < NQ; q++)
                acc[q] = fmul2(dup2(__fsub_rn(A.b, __fmul_rn(bdt, sm.par[lz * Sm::kParLayer + q * kParamStride + 6]))), f[q]);
        } else {
            const u64 kb = dup2(A.kb);
#pragma unroll
            for (int q = 0; q < NQ; q++)
                acc[q] = fmul2(kb, f[q]);
        }
        if (has_fn) {
            wait(bN);
            const u64 an = dup2(A.an);
#pragma unroll
            for (int q = 0; q < NQ; q++)
                acc[q] = ffma2(an, ld2(&pN[hf * NQ + q][c2]), acc[q]);
        }
        // f^n is consumed: the z-neighbour's slices land in its place
        __syncwarp();
        if (lane >= RZ && lane < RZ + N1) {
            const float *zs = csrc;
            const uint32_t bb = bar(bN);
            fence_proxy_async();
            if (lane == RZ)
                mbar_arrive_expect_tx(bb, zs ? kPart : 0);
            if (zs)
                bulk_g2s(part0 + bN * kBuf + (lane - RZ) * 2 * N1 * kRow, zs + vl * tstride, 2 * N1 * kRow, bb);
        }
        // The N1 lines of direction d of this half-warp (x- and y-lines of layer lz, z-lines of slice iy = lz):
        // line k has face point fp = k + N1 lz on both faces; fnode(j) its node j, nb its row in the staged
        // neighbour's part. lo: the tile's octant stages the low-side neighbour; es: that neighbour, < 0 on a
        // boundary face (its ghost value instead). Velocities whose flow enters through the other face take
        // that face's exterior trace, read for all lines of the direction at once and only where some
        // velocity of the warp needs it. Per half of a pair the operations and their order are those of
        // curv_line_c and trace_line.
        auto lines = [&](auto dc, bool lo, int es, auto load, auto nb, auto put) {
            constexpr int d = decltype(dc)::value;
            auto node = [&](int k, int j) {
                return d == 0 ? j + N1 * k + NQ * lz : (d == 1 ? k + N1 * j + NQ * lz : k + N1 * lz + NQ * j);
            };
            auto trace = [&](const u64(&v)[N1], bool lp) {  // trace_line with the weights lp or lm
                u64 t = 0;
#pragma unroll
                for (int j = 1; j < N1; j++)
                    t = ffma2(dup2(lp ? A.ops.lp[j] : A.ops.lm[j]), fsub2(v[j], v[0]), t);
                return fadd2(v[0], t);
            };
            // ghost value of every line on face g (the wall test is outside the loops: no load is formed from
            // a pointer that may be null)
            auto ghosts = [&](int g, u64(&o)[N1]) {
                const u64 gv = *reinterpret_cast<const u64 *>(A.ghost + (int64_t)g * A.nslots + slot);
                if (A.mesh.bc[g] == 2) {
                    const float *rw = A.rhow + ((int64_t)g * A.nfmax + face_elem(A.mesh, ec, d)) * NQ + N1 * lz;
#pragma unroll
                    for (int k = 0; k < N1; k++)
                        o[k] = fmul2(gv, dup2(__ldg(rw + k)));
                } else {
#pragma unroll
                    for (int k = 0; k < N1; k++)
                        o[k] = gv;
                }
            };
            float uL[N1][2], uR[N1][2];
            bool far = false;
#pragma unroll
            for (int k = 0; k < N1; k++) {
                const float4 nL = sm.fnm[d][0][k + N1 * lz], nR = sm.fnm[d][1][k + N1 * lz];
#pragma unroll
                for (int s = 0; s < 2; s++) {
                    uL[k][s] = fmaf(nL.z, x[2][s], fmaf(nL.y, x[1][s], nL.x * x[0][s]));
                    uR[k][s] = fmaf(nR.z, x[2][s], fmaf(nR.y, x[1][s], nR.x * x[0][s]));
                    far = far || (lo ? uR[k][s] < 0.f : uL[k][s] > 0.f);
                }
            }
            u64 tF[N1];  // the other side's trace
#pragma unroll
            for (int k = 0; k < N1; k++)
                tF[k] = 0;
            if (__any_sync(0xffffffffu, far)) {
                const int eo = upwind_neighbour(A.mesh, ec, d, !lo);
                if (!GEN || eo >= 0) {
                    const float *on = A.src + fidx(vl, eo, 0, c2, E, NP);
#pragma unroll
                    for (int k = 0; k < N1; k++) {
                        const bool need = lo ? uR[k][0] < 0.f || uR[k][1] < 0.f : uL[k][0] > 0.f || uL[k][1] > 0.f;
                        u64 v[N1];
#pragma unroll
                        for (int j = 0; j < N1; j++)
                            v[j] = need ? __ldg(reinterpret_cast<const u64 *>(on + node(k, j) * kWarp)) : 0;
                        tF[k] = trace(v, !lo);
                    }
                } else {
                    ghosts(2 * d + (lo ? 1 : 0), tF);
                }
            }
            // all lines of the direction together, constant by constant: an f32x2 instruction takes a
            // coefficient as a register pair, which then serves N1 lines instead of one
            u64 F[N1][N1], oL[N1], oR[N1], tS[N1], v0[N1];
#pragma unroll
            for (int j = 0; j < N1; j++)
#pragma unroll
                for (int k = 0; k < N1; k++) {
                    const u64 fl = load(k, j);
                    const float4 mt = sm.met[d][node(k, j)];
                    float u[2];
#pragma unroll
                    for (int s = 0; s < 2; s++)
                        u[s] = fmaf(mt.z, x[2][s], fmaf(mt.y, x[1][s], mt.x * x[0][s]));
                    F[k][j] = fmul2(pack2(u[0], u[1]), fl);
                    oL[k] = ffma2(dup2(A.ops.lm[j]), fl, j == 0 ? 0ull : oL[k]);
                    oR[k] = ffma2(dup2(A.ops.lp[j]), fl, j == 0 ? 0ull : oR[k]);
                }
            // the staged side's trace (trace_line)
#pragma unroll
            for (int j = 0; j < N1; j++) {
                const u64 c = dup2(lo ? A.ops.lp[j] : A.ops.lm[j]);
#pragma unroll
                for (int k = 0; k < N1; k++) {
                    if (j == 0)
                        v0[k] = nb(k, 0);
                    else
                        tS[k] = ffma2(c, fsub2(nb(k, j), v0[k]), j == 1 ? 0ull : tS[k]);
                }
            }
#pragma unroll
            for (int k = 0; k < N1; k++)
                tS[k] = fadd2(v0[k], tS[k]);
            if (GEN && es < 0)  // the staged side's ghost value of every line on a boundary face
                ghosts(2 * d + (lo ? 0 : 1), tS);
            // the common fluxes at both faces, over oL and oR
#pragma unroll
            for (int k = 0; k < N1; k++) {
                float tL2[2], tR2[2], oL2[2], oR2[2];
                unpack2(lo ? tS[k] : tF[k], tL2[0], tL2[1]);
                unpack2(lo ? tF[k] : tS[k], tR2[0], tR2[1]);
                unpack2(oL[k], oL2[0], oL2[1]);
                unpack2(oR[k], oR2[0], oR2[1]);
#pragma unroll
                for (int s = 0; s < 2; s++) {
                    oL2[s] = uL[k][s] * (uL[k][s] > 0.f ? tL2[s] : oL2[s]);
                    oR2[s] = uR[k][s] * (uR[k][s] < 0.f ? tR2[s] : oR2[s]);
                }
                oL[k] = pack2(oL2[0], oL2[1]);
                oR[k] = pack2(oR2[0], oR2[1]);
            }
#pragma unroll
            for (int i = 0; i < N1; i++) {
                u64 a[N1];
#pragma unroll
                for (int k = 0; k < N1; k++)
                    a[k] = ffma2(dup2(A.ops.gl[i]), oL[k], fmul2(dup2(A.ops.gr[i]), oR[k]));
#pragma unroll
                for (int j = 0; j < N1; j++) {
                    const u64 c = dup2(A.ops.DM[i][j]);
#pragma unroll
                    for (int k = 0; k < N1; k++)
                        a[k] = ffma2(c, F[k][j], a[k]);
                }
#pragma unroll
                for (int k = 0; k < N1; k++)
                    put(k, i, a[k]);
            }
        };
        // a += -b dt / J of the layer's node q times the line sum
        auto scale = [&](int q, u64 sum, u64 a) { return ffma2(dup2(sm.sj[q + NQ * lz]), sum, a); };
        wait(bX);
        lines(std::integral_constant<int, 0>{}, (oct & 1) != 0, en[0], [&](int k, int j) { return f[j + N1 * k]; },
              [&](int k, int j) { return ld2(&pX[j + N1 * k][c2]); },
              [&](int k, int j, u64 a) { acc[j + N1 * k] = scale(j + N1 * k, a, acc[j + N1 * k]); });
        wait(bY);
        lines(std::integral_constant<int, 1>{}, (oct & 2) != 0, en[1], [&](int k, int j) { return f[k + N1 * j]; },
              [&](int k, int j) { return ld2(&pY[k + N1 * j][c2]); },
              [&](int k, int j, u64 a) { acc[k + N1 * j] = scale(k + N1 * j, a, acc[k + N1 * j]); });
        // the x- and y-neighbours are consumed: the next tile's f_s and f^n land in their places
        __syncwarp();
        if (more && (lane == 0 || (lane == RFN && has_fn))) {
            fence_proxy_async();
            issue(csrc, vl + 1, lane == 0 ? bX : bY);
        }
        __syncthreads();  // B1: every layer of the element tile has landed (each warp waited for its own)
        // z-lines of slice iy = lz (all layers) from the shared tile, the upwind trace from the staged
        // neighbour rows; each line's derivative sums overwrite the rows it read
        wait(bN);
        lines(std::integral_constant<int, 2>{}, (oct & 4) != 0, en[2],
              [&](int k, int j) { return ld2(&F[k + N1 * lz + NQ * j][c2]); },
              [&](int k, int j) { return ld2(&pN[2 * N1 * j + N1 * hf + k][c2]); },
              [&](int k, int j, u64 a) { st2(&F[k + N1 * lz + NQ * j][c2], a); });
        // the z-neighbour is consumed: the next tile's x-neighbour lands in its place; warp 0 also brings the
        // next tile's velocity table into the other table buffer, which every warp is done with (B1)
        __syncwarp();
        if (more && (lane == RX || tid == RT)) {  // one code path for both role lanes
            const bool t = lane == RT;
            const float *xs = t ? nullptr : (turn ? role_src(enn) : csrc);
            const float *ns = t ? A.vtab + (int64_t)(vt + 1) * kTabRows * kWarp : (xs ? xs + (vl + 1) * tstride : nullptr);
            const uint32_t bb = t ? tbar(b ^ 1) : bar(bN);
            const uint32_t dst = t ? smem_u32(&sm.tab[b ^ 1][0][0]) : part0 + bN * kBuf;
            const uint32_t bytes = t ? kTabRows * kRow : kPart;
            fence_proxy_async();
            mbar_arrive_expect_tx(bb, ns ? bytes : 0);
            if (ns)
                bulk_g2s(dst, ns, bytes, bb);
        }
        __syncthreads();  // B2: z-sums complete
#pragma unroll
        for (int q = 0; q < NQ; q++)
            acc[q] = scale(q, ld2(&F[q + NQ * lz][c2]), acc[q]);
        __syncwarp();  // the z-sums of these layers are read before their rows take the stage output
        // BGK source towards the conservative Maxwellian, Shu-Osher combination, store
        float W0, W1;
        unpack2(ld2(&sm.tab[b][3][c2]), W0, W1);
        const float gm[2] = {W0 != 0.f ? 1.f : 0.f, W1 != 0.f ? 1.f : 0.f};  // the padding mask
        const bool iso = !GEN || A.viso;
        float xs[2], mm[3][2], mms[2];
#pragma unroll
        for (int s = 0; s < 2; s++) {
            xs[s] = x[0][s] * x[0][s] + x[1][s] * x[1][s] + x[2][s] * x[2][s];
#pragma unroll
            for (int d = 0; d < 3; d++)
                mm[d][s] = m[d][s] * m[d][s];
            mms[s] = mm[0][s] + mm[1][s] + mm[2][s];
            if (iso) {
                mm[0][s] = mm[1][s] = mms[s];
                mm[2][s] = 0.f;
            }
        }
        const u64 cg = pack2(A.kg * gm[0], A.kg * gm[1]), cf = pack2(bdt * gm[0], bdt * gm[1]);
        const u64 gm2 = pack2(gm[0], gm[1]);
        const u64 X0 = pack2(x[0][0], x[0][1]), X1 = pack2(x[1][0], x[1][1]), X2 = pack2(x[2][0], x[2][1]);
        const u64 XS = pack2(xs[0], xs[1]);
        float *dst = A.dst + fidx(vl, e, NQ * lz, c2, E, NP);
        u64 lsum = 0;  // limiter: this layer's weighted sum and minimum
        float lmin[2] = {3.4e38f, 3.4e38f};
        auto put_out = [&](int q, u64 o) {  // the stored value, and its transposed copy for the moments
            __stcs(reinterpret_cast<u64 *>(dst + q * kWarp), o);
            st2(&F[q + NQ * lz][c2 ^ (4 * ((q + (NQ % 8 ? NQ * hf : 0)) & 7))], o);  // (its row mod 8)
        };
        auto bgk_src = [&](auto vtau_c, auto force_c, auto lim_c) {
            constexpr bool VT = decltype(vtau_c)::value, FP = decltype(force_c)::value;
            constexpr bool LIM = decltype(lim_c)::value;
#pragma unroll
            for (int q = 0; q < NQ; q++) {
                const float4 *pp = reinterpret_cast<const float4 *>(&sm.par[lz * Sm::kParLayer + q * kParamStride]);
                const float4 pa = pp[0], pb = pp[1];  // (a, b_x, b_y, b_z), (p4, p5, p6, 2^x constant)
                float ex[2];
#pragma unroll
                for (int s = 0; s < 2; s++) {
                    const float lin = fmaf(pa.w, m[2][s], fmaf(pa.z, m[1][s], fmaf(pa.y, m[0][s], pa.x)));
                    ex[s] = GEN ? fmaf(pb.x, mm[0][s], fmaf(pb.y, mm[1][s], fmaf(pb.z, mm[2][s], lin)))
                                : fmaf(pb.x, mms[s], fmaf(pb.y, mms[s], lin));
                }
                float g[2];
                exp2_fp32x2(pack2(ex[0], ex[1]), dup2(pb.w), g[0], g[1]);
                u64 gc = cg;
                if constexpr (VT)  // kg = b - kb exactly, kb as in the accumulator above
                    gc = fmul2(dup2(__fsub_rn(A.b, __fsub_rn(A.b, __fmul_rn(bdt, pb.z)))), gm2);
                if constexpr (FP) {  // body-force source g (q0 + q . xi + q4 |xi|^2)
                    const float *fq = &sm.fpar[q + NQ * lz][0];
                    const float4 f4 = *reinterpret_cast<const float4 *>(fq);
                    const u64 qv = ffma2(dup2(fq[4]), XS,
                                         ffma2(dup2(f4.w), X2, ffma2(dup2(f4.z), X1, ffma2(dup2(f4.y), X0, dup2(f4.x)))));
                    gc = ffma2(cf, qv, gc);  // on top of the node's own Maxwellian weight
                }
                acc[q] = ffma2(gc, pack2(g[0], g[1]), acc[q]);
                if constexpr (LIM) {  // stored after the limiter below
                    lsum = ffma2(dup2(sm.wj[q + NQ * lz]), acc[q], lsum);
                    float o0, o1;
                    unpack2(acc[q], o0, o1);
                    lmin[0] = fminf(lmin[0], o0);
                    lmin[1] = fminf(lmin[1], o1);
                } else {
                    put_out(q, acc[q]);
                }
            }
        };
        using T_ = std::true_type;
        using F_ = std::false_type;
        if constexpr (GEN) {
            if (A.limiter) {
                if (A.fpar)
                    A.vtau ? bgk_src(T_{}, T_{}, T_{}) : bgk_src(F_{}, T_{}, T_{});
                else
                    A.vtau ? bgk_src(T_{}, F_{}, T_{}) : bgk_src(F_{}, F_{}, T_{});
            } else {
                if (A.fpar)
                    A.vtau ? bgk_src(T_{}, T_{}, F_{}) : bgk_src(F_{}, T_{}, F_{});
                else
                    A.vtau ? bgk_src(T_{}, F_{}, F_{}) : bgk_src(F_{}, F_{}, F_{});
            }
        } else {
            bgk_src(F_{}, F_{}, F_{});
        }
        if (GEN && A.limiter) {
            // Zhang-Shu (Sec. 2.1, Eqs. 10-11) over the physical element: weights W J over their sum
            st2(&sm.lim[0][lz][c2], lsum);
            st2(&sm.lim[1][lz][c2], pack2(lmin[0], lmin[1]));
            __syncthreads();  // B3 (the general form only)
            float mean[2] = {0.f, 0.f}, mn[2] = {sm.lim[1][0][c2], sm.lim[1][0][c2 + 1]}, beta[2];
#pragma unroll
            for (int s = 0; s < 2; s++) {
#pragma unroll
                for (int lw = 0; lw < N1; lw++) {
                    mean[s] += sm.lim[0][lw][c2 + s];
                    mn[s] = fminf(mn[s], sm.lim[1][lw][c2 + s]);
                }
                mean[s] *= sm.iwj;
                beta[s] = mn[s] < 0.f ? fminf(fabsf(mean[s] / (mean[s] - mn[s])), 1.f) : 1.f;
            }
            if (mn[0] < 0.f || mn[1] < 0.f) {
#pragma unroll
                for (int q = 0; q < NQ; q++) {
                    float o[2];
                    unpack2(acc[q], o[0], o[1]);
#pragma unroll
                    for (int s = 0; s < 2; s++)
                        o[s] = mn[s] < 0.f ? fmaf(beta[s], o[s] - mean[s], mean[s]) : o[s];
                    acc[q] = pack2(o[0], o[1]);
                }
            }
#pragma unroll
            for (int q = 0; q < NQ; q++)
                put_out(q, acc[q]);
        }
        // moments of these layers' nodes (Eq. 2 with Eq. 12) of the stored values
        __syncwarp();
        u64 pm[NR][5];
#pragma unroll
        for (int r = 0; r < NR; r++)
#pragma unroll
            for (int c = 0; c < 5; c++)
                pm[r][c] = 0ull;
#pragma unroll
        for (int k = 0; k < 8; k += 4) {
            const int kk = 8 * kg + k;
            u64 wv[5][2];
            {
                const float4 W4 = *reinterpret_cast<const float4 *>(&sm.tab[b][3][kk]);
                const float4 E4 = *reinterpret_cast<const float4 *>(&sm.tab[b][4][kk]);
                wv[0][0] = pack2(W4.x, W4.y);
                wv[0][1] = pack2(W4.z, W4.w);
                wv[4][0] = pack2(E4.x, E4.y);
                wv[4][1] = pack2(E4.z, E4.w);
#pragma unroll
                for (int d = 0; d < 3; d++) {  // W m_d: a power of two times an integer, exact
                    const float4 M4 = *reinterpret_cast<const float4 *>(&sm.tab[b][d][kk]);
                    wv[1 + d][0] = fmul2(pack2(W4.x, W4.y), pack2(M4.x, M4.y));
                    wv[1 + d][1] = fmul2(pack2(W4.z, W4.w), pack2(M4.z, M4.w));
                }
            }
#pragma unroll
            for (int r = 0; r < NR; r++) {
                const int row = lay + np + 8 * r;  // (row mod 8 = np)
                const float4 v = *reinterpret_cast<const float4 *>(&F[row][kk ^ (4 * np)]);
                const u64 v01 = pack2(v.x, v.y), v23 = pack2(v.z, v.w);
#pragma unroll
                for (int c = 0; c < 5; c++) {
                    pm[r][c] = ffma2(wv[c][0], v01, pm[r][c]);
                    pm[r][c] = ffma2(wv[c][1], v23, pm[r][c]);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < NR; r++)
#pragma unroll
            for (int c = 0; c < 5; c++)
                msum[r][c] += sum2(pm[r][c]);
        // this tile's f_s buffer is done with (the other warp's reads and writes of this part ended at B2): the
        // next tile's y-neighbour lands there
        __syncwarp();
        if (more && lane == RY) {
            const float *ys = turn ? role_src(enn) : csrc;
            fence_proxy_async();
            issue(ys, vl + 1, bF);
        }
        // the end of a moment group: combine the 4 velocity eighths of a row (in the tile loop, as it was first written;
        // outside it, as in k_stage3s, it was not measured here)
        if (vl + 1 == ge) {
            const int grp = moment_group(A, blockIdx.x / E, vl);
            ge = min(ge + A.G, vl1);
#pragma unroll
            for (int r = 0; r < NR; r++)
#pragma unroll
                for (int c = 0; c < 5; c++) {
                    float s = msum[r][c];
                    s += __shfl_xor_sync(0xffffffffu, s, 1);
                    s += __shfl_xor_sync(0xffffffffu, s, 2);
                    if (kg == 0)
                        A.partial[((int64_t)grp * 5 + c) * A.npts + (int64_t)e * NP + lay + np + 8 * r] = s;
                    msum[r][c] = 0.f;
                }
        }
#pragma unroll
        for (int d = 0; d < 3; d++)
            en[d] = enn[d];
        if (turn) {
            csrc = role_src(en);
            octc = octn;
        }
        const int t = bF;
        bF = bX;
        bX = bN;
        bN = bY;
        bY = t;
    }
}


template <int N1>
cudaError_t prepare3c()
{
    if constexpr (stage3c_pairs(N1)) {
        cudaError_t e = cudaFuncSetAttribute(k_stage3cp<N1, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)sizeof(Stage3cpSmem<N1, 0>));
        return e != cudaSuccess ? e : cudaFuncSetAttribute(k_stage3cp<N1, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                           (int)sizeof(Stage3cpSmem<N1, 1>));
    } else {
        cudaError_t e = cudaFuncSetAttribute(k_stage3c<N1, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)sizeof(Stage3cSmem<N1, 0>));
        return e != cudaSuccess ? e : cudaFuncSetAttribute(k_stage3c<N1, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                           (int)sizeof(Stage3cSmem<N1, 1>));
    }
}

template <int N1, int GEN>
cudaError_t launch3c(const StageArgs &A0, cudaStream_t s)
{
    StageArgs A = A0;
    if constexpr (stage3c_pairs(N1)) {
        using Sm = Stage3cpSmem<N1, GEN>;
        static_assert(offsetof(Sm, tab) % 16 == 0 && offsetof(Sm, par) % 16 == 0 && offsetof(Sm, met) % 16 == 0 &&
                          offsetof(Sm, fnm) % 16 == 0 && offsetof(Sm, fpar) % 16 == 0 && offsetof(Sm, lim) % 16 == 0 &&
                          offsetof(Sm, bar) % 8 == 0,
                      "8- and 16-byte shared accesses");
        plan_tasks(A, A.mesh.nelem, 152 * 16, 0.8, 0.5, 8);  // (12 free tiles: up to 1.24 of single groups' time)
        k_stage3cp<N1, GEN><<<A.mesh.nelem * A.ntasks, kWarp * N1 / 2, sizeof(Sm), s>>>(A);
    } else {
        plan_tasks(A, A.mesh.nelem, 152 * (N1 >= 4 ? BGK_STAGE3C_MINCTAS_P3 : 6), 0.8, 0.6);
        k_stage3c<N1, GEN><<<A.mesh.nelem * A.ntasks, kWarp * N1, sizeof(Stage3cSmem<N1, GEN>), s>>>(A);
    }
    return cudaGetLastError();
}

}  // namespace bgk
