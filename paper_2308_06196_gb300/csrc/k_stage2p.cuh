// k_stage2p.cuh -- the fused SSP-RK3 stage kernel of quadrilaterals of even line length (p = 1 and 3; FP32-split
// form) on packed pairs of velocities, every operand staged by bulk asynchronous copies; instantiated in
// k_stage2.cu.
#pragma once
#include <cstddef>
#include <type_traits>

#include "stage_common.cuh"

namespace bgk {

// ------------------------------------------------------------------------------------------------
// One warp per two consecutive elements: half-warp h holds element 2 b + h, lane l of it the velocities 2 l and
// 2 l + 1 of the tile, as k_stage3s (the halves of an f32x2 pair are two velocities of one node). All lines of
// an element are the half-warp's own registers, so no warp waits for another. Four buffers of
// the two elements rotate, each refilled as soon as it is consumed:
//   f_s    read into registers first, then the transposed output for the moment sums, then the next tile's
//          y-neighbour;    f^n    read next, then the next tile's x-neighbour;
//   the x-upwind neighbour, then the next tile's f_s;    the y-upwind neighbour, then the next tile's f^n.
// Every copy has a role lane (operand and half) that announces and issues its bytes on the buffer's barrier.
// Bound: latency and issue at 12 warps per SM. With a lane per velocity (k_stage2) the exponents alone returned
// 8 of the 24 cycles of shared-memory data per 32 degrees of freedom, and the neighbour lines came from L2
// lane by lane: 128^2 elements at p = 3, 32^2 velocities 0.174 -> 0.154 ms per octant launch (4.6 TB/s); 128 x
// 127 at p = 1, 40^2 velocities, three steps 5.72 -> 3.75 ms.
// Forms: GEN = 0 every face periodic, no limiter, constant tau, one velocity spacing; GEN = 1 everything.
// ------------------------------------------------------------------------------------------------
template <int N1, int GEN>
struct Stage2pSmem {
    static constexpr int NQ = N1 * N1;
    static constexpr int kParElem = NQ * kParamStride + 8;  // floats between the two elements' exponents
    // every member is read or written in 8- or 16-byte units
    alignas(16) float buf[4][2 * NQ][kWarp];
    alignas(16) float tab[2][5][kWarp];
    alignas(16) float par[2 * kParElem];
    unsigned long long bar[4];   // per buffer (two arrivals: one per half)
    unsigned long long tbar[2];  // the velocity tables
};

// warps (independent pairs of elements) per CTA, so that the kilobyte which a CTA reserves does not cost the
// twelfth warp; resident warps per SM that the registers are sized for
template <int N1>
constexpr int kStage2pWarps = N1 == 4 ? 2 : 4;
template <int N1>
constexpr int kStage2pResident = N1 == 4 ? 12 : 16;

template <int N1, int OCT, int GEN>
__global__ void __launch_bounds__(kWarp *kStage2pWarps<N1>, kStage2pResident<N1> / kStage2pWarps<N1>)
    k_stage2p(const StageArgs A)
{
    using u64 = unsigned long long;
    constexpr int NQ = N1 * N1;
    constexpr uint32_t kRow = kWarp * sizeof(float);
    using Sm = Stage2pSmem<N1, GEN>;
    extern __shared__ __align__(16) unsigned char smraw[];
    Sm &sm = reinterpret_cast<Sm *>(smraw)[threadIdx.x >> 5];

    const int lane = threadIdx.x & 31, hf = lane >> 4, c2 = 2 * (lane & 15);
    const int E = A.mesh.nelem, EB = (E + 1) / 2;
    const int unit = blockIdx.x * kStage2pWarps<N1> + (threadIdx.x >> 5), eb = 2 * (unit % EB);
    if (unit >= EB * A.ntasks)  // no barrier below involves other warps
        return;
    int vl0, vl1;
    task_tiles(A, unit / EB, vl0, vl1);
    int ge = min(vl0 + A.G, vl1);  // end of the moment group
    const int e = min(eb + hf, E - 1);  // (an odd count's last half repeats the last element and stores nothing)
    const bool real = eb + hf < E;
    const int row0 = NQ * hf;  // this half's first row

    for (int q = lane; q < 2 * NQ * kParamStride / 4; q += kWarp) {
        constexpr int kQ4 = NQ * kParamStride / 4;
        const int el = min(eb + q / kQ4, E - 1);
        *reinterpret_cast<float4 *>(&sm.par[(q / kQ4) * Sm::kParElem + 4 * (q % kQ4)]) =
            __ldg(reinterpret_cast<const float4 *>(A.param + (int64_t)el * NQ * kParamStride) + q % kQ4);
    }
    const uint32_t bar0 = smem_u32(&sm.bar[0]), tbar0 = smem_u32(&sm.tbar[0]);
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    auto tbar = [&](int b) { return tbar0 + 8u * (uint32_t)b; };
    if (lane == 0) {
#pragma unroll
        for (int i = 0; i < 4; i++)
            mbar_init(bar(i), 2);
        mbar_init(tbar(0), 1);
        mbar_init(tbar(1), 1);
        fence_mbar_init();
    }
    __syncwarp();

    const bool has_fn = A.fn != nullptr;
    // role lanes 2 op + half, op = 0 f_s, 1 f^n, 2 / 3 the x- / y-neighbour; lane 8 the velocity table
    const int op = lane >> 1;
    const bool role = lane < 8;
    const int er = min(eb + (lane & 1), E - 1);  // a role lane's element
    const int erc[3] = {er % A.mesh.ne[0], er / A.mesh.ne[0], 0};
    const int64_t tstride = (int64_t)E * NQ * kWarp;
    auto role_src = [&](int oct) -> const float * {  // the copy's source at tile 0, null at a boundary face
        if (op == 0)
            return A.src + fidx(0, er, 0, 0, E, NQ);
        if (op == 1)
            return A.fn + fidx(0, er, 0, 0, E, NQ);
        const int n = upwind_neighbour(A.mesh, erc, op - 2, ((oct >> (op - 2)) & 1) != 0);
        return n >= 0 ? A.src + fidx(0, n, 0, 0, E, NQ) : nullptr;
    };
    const uint32_t part0 = smem_u32(&sm.buf[0][NQ * (lane & 1)][0]);  // a role lane's half of buffer 0
    constexpr uint32_t kBuf = 2 * NQ * kRow, kPart = NQ * kRow;
    auto issue = [&](const float *from, int vl, int k) {
        mbar_arrive_expect_tx(bar(k), from ? kPart : 0);
        if (from)
            bulk_g2s(part0 + k * kBuf, from + vl * tstride, kPart, bar(k));
    };
    int octc = OCT < 8 ? OCT : (int)__ldg(A.toct + A.vt0 + vl0);
    const float *csrc = role ? role_src(octc) : nullptr;
    const int ec[3] = {e % A.mesh.ne[0], e / A.mesh.ne[0], 0};
    int enx = upwind_neighbour(A.mesh, ec, 0, (octc & 1) != 0), eny = upwind_neighbour(A.mesh, ec, 1, (octc & 2) != 0);
    int bF = 0, bN = 1, bX = 2, bY = 3;
    if (role && (op != 1 || has_fn))
        issue(csrc, vl0, op == 0 ? bF : (op == 1 ? bN : (op == 2 ? bX : bY)));
    auto issue_table = [&](int vl, int b) {  // lane 8
        mbar_arrive_expect_tx(tbar(b), 5 * kRow);
        bulk_g2s(smem_u32(&sm.tab[b][0][0]), A.vtab + (int64_t)(A.vt0 + vl) * 5 * kWarp, 5 * kRow, tbar(b));
    };
    if (lane == 8)
        issue_table(vl0, 0);
    uint32_t ph = 0;  // phase parity, bit i for bar(i), bit 4 + b for tbar(b)
    auto wait = [&](int i) {
        mbar_wait(bar(i), (ph >> i) & 1, A.err);
        ph ^= 1u << i;
    };

    // moment sums: lane = (row np + 8 r of the 2 NQ rows, np = lane / 4) x (velocity eighth kg = lane % 4)
    const int np = lane >> 2, kg = lane & 3;
    constexpr int NR = 2 * NQ / 8;
    float msum[NR][5];
#pragma unroll
    for (int r = 0; r < NR; r++)
#pragma unroll
        for (int c = 0; c < 5; c++)
            msum[r][c] = 0.f;
    const float bdt = A.b * A.dt;
    auto ld2 = [](const float *p) { return *reinterpret_cast<const u64 *>(p); };
    auto st2 = [](float *p, u64 v) { *reinterpret_cast<u64 *>(p) = v; };

    for (int vl = vl0; vl < vl1;) {  // a moment group
        for (; vl < ge; vl++) {
            const int vt = A.vt0 + vl;
            const int b = (vl - vl0) & 1;
            const bool more = vl + 1 < vl1;
            const int oct = octc, octn = OCT < 8 ? OCT : (more ? (int)__ldg(A.toct + vt + 1) : octc);
            const bool turn = OCT == 8 && octn != oct;
            const float *nsrc = csrc;  // this role lane's source of the next tile
            if (turn && role)
                nsrc = role_src(octn);
            float(*const F)[kWarp] = sm.buf[bF];
            const float(*const pN)[kWarp] = sm.buf[bN] + row0, (*const pX)[kWarp] = sm.buf[bX] + row0,
                             (*const pY)[kWarp] = sm.buf[bY] + row0;
            wait(bF);
            mbar_wait(tbar(b), (ph >> (4 + b)) & 1, A.err);
            ph ^= 1u << (4 + b);
            float m[3][2], x[2][2];
            u64 cdir[2];
#pragma unroll
            for (int d = 0; d < 3; d++)
                unpack2(ld2(&sm.tab[b][d][c2]), m[d][0], m[d][1]);
#pragma unroll
            for (int d = 0; d < 2; d++) {
#pragma unroll
                for (int s = 0; s < 2; s++)
                    x[d][s] = fmaf(A.vs[d], m[d][s], A.vc[d]);
                cdir[d] = pack2(-A.mesh.inv_h2[d] * x[d][0] * bdt, -A.mesh.inv_h2[d] * x[d][1] * bdt);
            }
            u64 f[NQ], acc[NQ];
#pragma unroll
            for (int q = 0; q < NQ; q++)
                f[q] = ld2(&F[row0 + q][c2]);
            // acc = an f^n + b (1 - dt/tau) f_s
            if (GEN && A.vtau) {
#pragma unroll
                for (int q = 0; q < NQ; q++)
                    acc[q] = fmul2(dup2(__fsub_rn(A.b, __fmul_rn(bdt, sm.par[hf * Sm::kParElem + q * kParamStride + 6]))), f[q]);
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
                    acc[q] = ffma2(an, ld2(&pN[q][c2]), acc[q]);
            }
            __syncwarp();  // f^n is consumed: the next tile's x-neighbour; the other table buffer: its table
            if (more && ((role && op == 2) || lane == 8)) {
                fence_proxy_async();
                if (lane == 8)
                    issue_table(vl + 1, b ^ 1);
                else
                    issue(nsrc, vl + 1, bN);
            }
            // The lines of one direction: line k's nodes f[line(k, j)], its upwind neighbour's row nb(k, j); where
            // that is no element (a Dirichlet ghost) the jump is the ghost's
            auto lines = [&](auto dc, int en, const float(*nbr)[kWarp], auto row) {
                constexpr int d = decltype(dc)::value;
                const bool left = (oct >> d) & 1, inner = GEN == 0 || en >= 0;
                u64 gh = 0;
                if (GEN && !inner)
                    gh = *reinterpret_cast<const u64 *>(A.ghost + (2 * d + (left ? 0 : 1)) * A.nslots + vt * kWarp + c2);
#pragma unroll
                for (int k = 0; k < N1; k++) {
                    u64 fl[N1], sv[N1], v[N1];
#pragma unroll
                    for (int j = 0; j < N1; j++) {
                        fl[j] = f[row(k, j)];
                        v[j] = ld2(&nbr[row(k, j)][c2]);
                    }
                    auto side = [&](auto left_c) {
                        constexpr bool LEFT = decltype(left_c)::value;
                        constexpr int R = LEFT ? 0 : N1 - 1;
                        const u64 tj = trace_jump2<N1, LEFT>(v, fl[R], A.ops);
                        const u64 tr = GEN == 0 ? tj : (inner ? tj : fsub2(gh, fl[R]));  // (per element: a select)
                        line_sums_jump2<N1, LEFT>(sv, fl, tr, A.ops);
                    };
                    if (left)
                        side(std::true_type{});
                    else
                        side(std::false_type{});
#pragma unroll
                    for (int j = 0; j < N1; j++)
                        acc[row(k, j)] = ffma2(cdir[d], sv[j], acc[row(k, j)]);
                }
            };
            wait(bX);
            lines(std::integral_constant<int, 0>{}, enx, pX, [](int k, int j) { return j + N1 * k; });
            __syncwarp();  // the x-neighbour is consumed: the next tile's f_s
            if (more && role && op == 0) {
                fence_proxy_async();
                issue(csrc, vl + 1, bX);
            }
            wait(bY);
            lines(std::integral_constant<int, 1>{}, eny, pY, [](int k, int j) { return k + N1 * j; });
            __syncwarp();  // the y-neighbour is consumed: the next tile's f^n
            if (more && has_fn && role && op == 1) {
                fence_proxy_async();
                issue(csrc, vl + 1, bY);
            }
            // BGK source towards the conservative Maxwellian, Shu-Osher combination, store
            float W0, W1;
            unpack2(ld2(&sm.tab[b][3][c2]), W0, W1);
            const float gm[2] = {W0 != 0.f ? 1.f : 0.f, W1 != 0.f ? 1.f : 0.f};  // the padding mask
            const bool iso = !GEN || A.viso;
            float mm[3][2], mms[2];
#pragma unroll
            for (int s = 0; s < 2; s++) {
#pragma unroll
                for (int d = 0; d < 3; d++)
                    mm[d][s] = m[d][s] * m[d][s];
                mms[s] = mm[0][s] + mm[1][s] + mm[2][s];
                if (iso) {
                    mm[0][s] = mm[1][s] = mms[s];
                    mm[2][s] = 0.f;
                }
            }
            const u64 cg = pack2(A.kg * gm[0], A.kg * gm[1]), gm2 = pack2(gm[0], gm[1]);
            float *dst = A.dst + fidx(vl, e, 0, c2, E, NQ);
            auto put_out = [&](int q, u64 o) {  // the stored value, and its transposed copy for the moments
                if (real)
                    __stcs(reinterpret_cast<u64 *>(dst + q * kWarp), o);
                st2(&F[row0 + q][c2 ^ (4 * ((q + (NQ % 8 ? NQ * hf : 0)) & 7))], o);  // (its row mod 8)
            };
            __syncwarp();  // every lane has read its rows of F
            auto bgk_src = [&](auto vtau_c, auto lim_c) {
                constexpr bool VT = decltype(vtau_c)::value, LIM = decltype(lim_c)::value;
#pragma unroll
                for (int q = 0; q < NQ; q++) {
                    const float4 *pp = reinterpret_cast<const float4 *>(&sm.par[hf * Sm::kParElem + q * kParamStride]);
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
                    acc[q] = ffma2(gc, pack2(g[0], g[1]), acc[q]);
                    if constexpr (!LIM)
                        put_out(q, acc[q]);
                }
            };
            using T_ = std::true_type;
            using F_ = std::false_type;
            if constexpr (GEN) {
                if (A.limiter)
                    A.vtau ? bgk_src(T_{}, T_{}) : bgk_src(F_{}, T_{});
                else
                    A.vtau ? bgk_src(T_{}, F_{}) : bgk_src(F_{}, F_{});
            } else {
                bgk_src(F_{}, F_{});
            }
            if (GEN && A.limiter) {
                // Zhang-Shu (Sec. 2.1, Eqs. 10-11): the element mean (tensor Gauss-Legendre weights / 4, summing to
                // 1) and minimum of each velocity, all in this lane's registers
                u64 mean2 = 0;
                float mn[2] = {3.4e38f, 3.4e38f}, mean[2];
#pragma unroll
                for (int q = 0; q < NQ; q++) {
                    mean2 = ffma2(dup2(A.ops.wq[q % N1] * A.ops.wq[q / N1]), acc[q], mean2);
                    float o[2];
                    unpack2(acc[q], o[0], o[1]);
                    mn[0] = fminf(mn[0], o[0]);
                    mn[1] = fminf(mn[1], o[1]);
                }
                unpack2(mean2, mean[0], mean[1]);
                float beta[2];
#pragma unroll
                for (int s = 0; s < 2; s++)
                    beta[s] = fminf(fabsf(mean[s] / (mean[s] - mn[s])), 1.f);
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
            // moments of the elements' nodes (Eq. 2 with Eq. 12) of the stored values
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
                    const int row = np + 8 * r;  // (row mod 8 = np)
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
            __syncwarp();  // this tile's f_s buffer is done with: the next tile's y-neighbour
            if (more && role && op == 3) {
                fence_proxy_async();
                issue(nsrc, vl + 1, bF);
            }
            if (turn) {
                csrc = nsrc;
                octc = octn;
                enx = upwind_neighbour(A.mesh, ec, 0, (octc & 1) != 0);
                eny = upwind_neighbour(A.mesh, ec, 1, (octc & 2) != 0);
            }
            const int t = bF;
            bF = bX;
            bX = bN;
            bN = bY;
            bY = t;
        }
        // the end of a moment group: combine the 4 velocity eighths of a row
        const int grp = moment_group(A, unit / EB, vl - 1);
        ge = min(ge + A.G, vl1);
#pragma unroll
        for (int r = 0; r < NR; r++)
#pragma unroll
            for (int c = 0; c < 5; c++) {
                float s = msum[r][c];
                s += __shfl_xor_sync(0xffffffffu, s, 1);
                s += __shfl_xor_sync(0xffffffffu, s, 2);
                const int row = np + 8 * r;  // rows of the repeated half of an odd count: not stored
                if (kg == 0 && eb + row / NQ < E)
                    A.partial[((int64_t)grp * 5 + c) * A.npts + (int64_t)eb * NQ + row] = s;
                msum[r][c] = 0.f;
            }
    }
}

template <int N1, int OCT, int GEN>
cudaError_t launch2p(const StageArgs &A0, cudaStream_t s)
{
    using Sm = Stage2pSmem<N1, GEN>;
    static_assert(offsetof(Sm, tab) % 16 == 0 && offsetof(Sm, par) % 16 == 0 && offsetof(Sm, bar) % 8 == 0,
                  "8- and 16-byte shared accesses");
    constexpr int WP = kStage2pWarps<N1>;
    static_assert(sizeof(Sm) % 16 == 0 && WP * sizeof(Sm) <= 48 * 1024, "the default dynamic shared memory");
    StageArgs A = A0;
    const int EB = (A.mesh.nelem + 1) / 2;
    plan_tasks(A, EB, 152 * kStage2pResident<N1>, 0.8, 0.75);
    k_stage2p<N1, OCT, GEN><<<(EB * A.ntasks + WP - 1) / WP, kWarp * WP, WP * sizeof(Sm), s>>>(A);
    return cudaGetLastError();
}

}  // namespace bgk
