// k_stage3s.cuh -- the fused SSP-RK3 stage kernel for affine hexahedra of even line length (p = 3; FP32-split
// form) with every operand staged in shared memory by bulk asynchronous copies; instantiated in
// k_stage3_p3.cu.
#pragma once
#include <cstddef>
#include <type_traits>

#include "stage_common.cuh"


namespace bgk {

// ------------------------------------------------------------------------------------------------
// One CTA per (element, run of velocity tiles), one warp per two z-layers of the element's nodes: half-warp
// h of warp w holds layer 2 w + h, lane l of it the velocities 2 l and 2 l + 1 of the tile. Every value of a
// lane is then a pair in one 64-bit register (one 8-byte load), and the line sums, traces, relaxation and
// the 2^x run on packed FP32 pairs (f32x2) whose halves are two velocities of one node: no register is
// moved to form a pair, and an instruction covers 64 degrees of freedom. Each half performs the scalar
// form's operations in its order.
// Bound: the latency of the dependent FP32 pairs and shared loads at 12 warps per SM (issue slots half used),
// with shared memory's data path close behind: per 32 degrees of freedom it takes 19.5 cycles for the copies
// in (5), the lines (8), the exponents (4: a load returns 128 bytes per cycle, broadcast or not) and the
// moments (2.5) of the 27 that a launch takes. A lane per velocity with packed pairs of lines (four warps
// per element) read the exponents once per 32 velocities (8 cycles) and took 70 instructions per 32 degrees
// of freedom, now 52. 16^3 elements, 24^3 velocities: 1.265 ms per octant launch before (3.8 TB/s), now
// 1.108 (4.4 TB/s); with the limiter and a variable collision time (7 x 9 x 5 elements, 21^3) 0.102 -> 0.093.
// Every warp streams its own rows through shared memory with bulk asynchronous copies completed on the
// warp's own mbarriers:
// four buffers of the element whose roles rotate, each refilled as soon as it is consumed, so that every copy
// is issued between a quarter and all of a tile ahead of its use:
//   f_s    read into registers first; after the first block barrier the z-lines read the other layers' rows
//          and write their derivative sums back over the rows they read; the stage output is then
//          transposed through the warp's own rows for the moment sums; then the next tile's y-neighbour;
//   f^n    read first, then the z-upwind neighbour's rows of the warp's z-line slices, then the next tile's
//          x-neighbour;
//   the x-upwind neighbour, then the next tile's f_s;  the y-upwind neighbour, then the next tile's f^n.
// Four buffers of 8 KB leave 6 CTAs per SM where five (f_s double-buffered) left 5: two steps of the 16^3
// elements 63.3 -> 58.0 ms.
// Warp 0 also brings the tile's velocity table into a double-buffered block with a barrier of its own, which
// every warp waits on. No global load is left in the tile loop of the periodic form.
// A CTA runs R moment groups of G tiles and writes its running moment sums out after each (plan_tasks).
// ------------------------------------------------------------------------------------------------
// velocity table rows per tile: the grid indices m_x, m_y, m_z, the index-basis weight W (0 on padded
// slots) and the energy weight W sum_d r_d m_d^2; the moment weights W m_d are formed from them (exact)
constexpr int kTabRows = 5;

// Forms: GEN = 0 every face periodic or an exchange face, no force, no limiter, constant tau, one velocity
// spacing; GEN = 1 everything but the force source; GEN = 2 with the force source, whose polynomials take 2 KB
// of shared memory. CTAs per SM that the register allocation is sized for and shared memory allows:
template <int GEN>
constexpr int kStage3sCtas = GEN == 2 ? 5 : 6;

template <int N1, int GEN>
struct Stage3sSmem {
    static_assert(N1 % 2 == 0, "a warp holds two layers");
    static constexpr int NP = N1 * N1 * N1, NQ = N1 * N1, NW = N1 / 2;
    // floats between the exponents of consecutive layers: 16 bytes of bank offset between the two halves
    static constexpr int kParLayer = NQ * kParamStride + 8;
    // every member is read or written in 8- or 16-byte units
    alignas(16) float buf[4][NP][kWarp];  // the four rotating operands; warp w's part: rows 2 NQ w ..
    alignas(16) float tab[2][kTabRows][kWarp];
    alignas(16) float par[N1 * kParLayer];  // BGK exponents [layer][node][8]
    alignas(16) float fpar[GEN == 2 ? NP : 1][GEN == 2 ? kParamStride : 1];  // force polynomials
    alignas(16) float lim[GEN ? 2 : 1][GEN ? N1 : 1][GEN ? kWarp : 1];
    unsigned long long bar[NW][4];  // per warp and buffer
    unsigned long long tbar[2];     // the velocity tables' buffers
};

template <int N1, int OCT, int GEN>
__global__ void __launch_bounds__(kWarp *N1 / 2, kStage3sCtas<GEN>)
    k_stage3s(const StageArgs A)
{
    using u64 = unsigned long long;
    constexpr int NQ = N1 * N1;
    constexpr int NP = NQ * N1;
    constexpr int NW = N1 / 2;
    constexpr int NT = kWarp * NW;
    constexpr uint32_t kRow = kWarp * sizeof(float);  // one node's row of a tile: 128 bytes
    using Sm = Stage3sSmem<N1, GEN>;
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

    // per-point BGK exponents (and force polynomials) of the element
    {
        const float4 *src = reinterpret_cast<const float4 *>(A.param + (int64_t)e * NP * kParamStride);
        constexpr int kQ4 = NQ * kParamStride / 4;  // float4s of a layer
        for (int q = tid; q < N1 * kQ4; q += NT)
            *reinterpret_cast<float4 *>(&sm.par[(q / kQ4) * Sm::kParLayer + 4 * (q % kQ4)]) = __ldg(src + q);
        if (GEN == 2) {
            const float4 *f4 = reinterpret_cast<const float4 *>(A.fpar + (int64_t)e * NP * kParamStride);
            float4 *d4 = reinterpret_cast<float4 *>(&sm.fpar[0][0]);
            for (int q = tid; q < NP * kParamStride / 4; q += NT)
                d4[q] = __ldg(f4 + q);
        }
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
    // upwind neighbours of tile vl (one-octant launches: the same for the whole task), -1 on a
    // Dirichlet or wall face
    auto nbrs = [&](int vl, int (&en)[3]) {
        const int oct = OCT < 8 ? OCT : (int)__ldg(A.toct + A.vt0 + vl);
#pragma unroll
        for (int d = 0; d < 3; d++)
            en[d] = upwind_neighbour(A.mesh, ec, d, ((oct >> d) & 1) != 0);
    };
    // Bulk copies. Each copy of a tile has a role lane, so that the copies of one issue point cost the
    // warp one short code path: lane 0 the warp's f_s layers, lanes RZ .. RZ + N1 - 1 the z-upwind
    // neighbour's row groups j = lane - RZ of the warp's z-line slices (rows ix + N1 (2 w + h) + NQ j, landing
    // as ix + N1 h + 2 N1 j), lane RFN the warp's layers of f^n, lanes RX and RY the x- and y-upwind
    // neighbours' layers; lane RT of warp 0 the tile's velocity table. A role lane keeps the source of its
    // copy at tile 0 and adds the tile stride; a boundary face (no neighbour) gives only the barrier's
    // arrival. Across an exchange face the x-upwind neighbour is the element of the face's halo (the
    // neighbouring subdomain's layer, [tile][face element][node][lane]), whose tiles are eface elements apart.
    constexpr int RZ = 1, RFN = N1 + 1, RX = N1 + 2, RY = N1 + 3, RT = N1 + 4;
    const int64_t tstride = (int64_t)E * NP * kWarp;  // floats between consecutive tiles of one element
    const int64_t hstride = (int64_t)A.eface * NP * kWarp;
    const int lay = 2 * NQ * w;  // the warp's first row
    int64_t cstride = tstride;   // this lane's stride (hstride for a halo source)
    auto role_src = [&](const int (&en)[3], int oct) -> const float * {
        cstride = tstride;
        if (lane == RX && en[0] == kHaloNeighbour) {
            cstride = hstride;
            const int64_t r = ec[1] + (int64_t)A.mesh.ne[1] * ec[2];
            return A.halo[(oct & 1) ? 0 : 1] + (((int64_t)A.vt0 * A.eface + r) * NP + lay) * kWarp;
        }
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
            bulk_g2s(part0 + k * kBuf, from + vl * cstride, kPart, bb);
    };

    int en[3];
    nbrs(vl0, en);
    const float *csrc = role_src(en, OCT < 8 ? OCT : (int)__ldg(A.toct + A.vt0 + vl0));  // at tile 0
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
    const float bdt = A.b * A.dt;
    auto ld2 = [](const float *p) { return *reinterpret_cast<const u64 *>(p); };
    auto st2 = [](float *p, u64 v) { *reinterpret_cast<u64 *>(p) = v; };

    for (int vl = vl0; vl < vl1;) {  // a moment group
        for (; vl < ge; vl++) {
            const int vt = A.vt0 + vl;
            const int slot = vt * kWarp + c2;
            const int b = (vl - vl0) & 1;
            float(*const F)[kWarp] = sm.buf[bF];  // f_s, then the z-sums, then the output
            const float(*const pN)[kWarp] = sm.buf[bN] + lay, (*const pX)[kWarp] = sm.buf[bX] + lay + hf * NQ,
                             (*const pY)[kWarp] = sm.buf[bY] + lay + hf * NQ;
            int enn[3] = {en[0], en[1], en[2]};  // the next tile's neighbours
            if (OCT == 8 && vl + 1 < vl1)
                nbrs(vl + 1, enn);
            const bool more = vl + 1 < vl1;
            const int oct = OCT < 8 ? OCT : (int)__ldg(A.toct + vt);
            const bool l0 = (oct & 1) != 0, l1 = (oct & 2) != 0, l2 = (oct & 4) != 0;
            const int enx = en[0], eny = en[1], enz = en[2];

            wait(bF);
            mbar_wait(tbar(b), (ph >> (4 + b)) & 1, A.err);
            ph ^= 1u << (4 + b);
            // the two velocities: grid indices, velocities, advection factors
            float m[3][2], x[3][2];
            u64 cdir[3];
#pragma unroll
            for (int d = 0; d < 3; d++) {
                unpack2(ld2(&sm.tab[b][d][c2]), m[d][0], m[d][1]);
#pragma unroll
                for (int s = 0; s < 2; s++)
                    x[d][s] = fmaf(A.vs[d], m[d][s], A.vc[d]);
                cdir[d] = pack2(-A.mesh.inv_h2[d] * x[d][0] * bdt, -A.mesh.inv_h2[d] * x[d][1] * bdt);
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
                const float *zs = OCT < 8 ? csrc : role_src(en, oct);
                const uint32_t bb = bar(bN);
                fence_proxy_async();
                if (lane == RZ)
                    mbar_arrive_expect_tx(bb, zs ? kPart : 0);
                if (zs)
                    bulk_g2s(part0 + bN * kBuf + (lane - RZ) * 2 * N1 * kRow, zs + vl * tstride, 2 * N1 * kRow, bb);
            }
            // upwind value on a non-periodic face: the Dirichlet ghost Maxwellian, or the diffuse-wall
            // Maxwellian scaled by the wall density of the face point (face point of every line of this
            // half-warp: its index + N1 * lz)
            const int fx = 0 + (l0 ? 0 : 1), fy = 2 + (l1 ? 0 : 1), fz = 4 + (l2 ? 0 : 1);
            u64 gx = 0, gy = 0, gz = 0;
            const float *rwx = nullptr, *rwy = nullptr, *rwz = nullptr;
            if (GEN) {
                auto ghost = [&](int fc) { return *reinterpret_cast<const u64 *>(A.ghost + fc * A.nslots + slot); };
                gx = enx != -1 ? 0 : ghost(fx);
                gy = eny >= 0 ? 0 : ghost(fy);
                gz = enz >= 0 ? 0 : ghost(fz);
                if (enx < 0 && A.mesh.bc[fx] == 2)
                    rwx = A.rhow + ((int64_t)fx * A.nfmax + face_elem(A.mesh, ec, 0)) * NQ + N1 * lz;
                if (eny < 0 && A.mesh.bc[fy] == 2)
                    rwy = A.rhow + ((int64_t)fy * A.nfmax + face_elem(A.mesh, ec, 1)) * NQ + N1 * lz;
                if (enz < 0 && A.mesh.bc[fz] == 2)
                    rwz = A.rhow + ((int64_t)fz * A.nfmax + face_elem(A.mesh, ec, 2)) * NQ + N1 * lz;
            }
            // The N1 lines of this half-warp in one direction: line k's nodes line(k, j), its upwind neighbour's
            // row at nb(k, j); where that is no element (a Dirichlet or wall ghost) the jump is the ghost's
            auto lines = [&](bool left, bool inner, u64 gh, const float *rwp, auto line, auto nb, auto put) {
                float rw[N1];
                if (GEN && !inner) {
#pragma unroll
                    for (int k = 0; k < N1; k++)
                        rw[k] = rwp ? 0.f : 1.f;
                    if (rwp) {
#pragma unroll
                        for (int k = 0; k < N1; k++)
                            rw[k] = __ldg(rwp + k);
                    }
                }
#pragma unroll
                for (int k = 0; k < N1; k++) {
                    u64 fl[N1], sv[N1], v[N1];
#pragma unroll
                    for (int j = 0; j < N1; j++) {
                        fl[j] = line(k, j);
                        v[j] = nb(k, j);
                    }
                    auto side = [&](auto left_c) {
                        constexpr bool LEFT = decltype(left_c)::value;
                        constexpr int R = LEFT ? 0 : N1 - 1;
                        const u64 tr = GEN == 0 || inner ? trace_jump2<N1, LEFT>(v, fl[R], A.ops)
                                                         : ffma2(gh, dup2(rw[k]), fmul2(dup2(-1.f), fl[R]));
                        line_sums_jump2<N1, LEFT>(sv, fl, tr, A.ops);
                    };
                    if (left)
                        side(std::true_type{});
                    else
                        side(std::false_type{});
#pragma unroll
                    for (int j = 0; j < N1; j++)
                        put(k, j, sv[j]);
                }
            };
            wait(bX);
            lines(l0, enx != -1, gx, rwx, [&](int k, int j) { return f[j + N1 * k]; },
                  [&](int k, int j) { return ld2(&pX[j + N1 * k][c2]); },
                  [&](int k, int j, u64 s) { acc[j + N1 * k] = ffma2(cdir[0], s, acc[j + N1 * k]); });
            wait(bY);
            lines(l1, eny >= 0, gy, rwy, [&](int k, int j) { return f[k + N1 * j]; },
                  [&](int k, int j) { return ld2(&pY[k + N1 * j][c2]); },
                  [&](int k, int j, u64 s) { acc[k + N1 * j] = ffma2(cdir[1], s, acc[k + N1 * j]); });
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
            lines(l2, enz >= 0, gz, rwz, [&](int k, int j) { return ld2(&F[k + N1 * lz + NQ * j][c2]); },
                  [&](int k, int j) { return ld2(&pN[2 * N1 * j + N1 * hf + k][c2]); },
                  [&](int k, int j, u64 s) { st2(&F[k + N1 * lz + NQ * j][c2], s); });
            // the z-neighbour is consumed: the next tile's x-neighbour lands in its place; warp 0 also brings the
            // next tile's velocity table into the other table buffer, which every warp is done with (B1)
            __syncwarp();
            if (more && (lane == RX || tid == RT)) {  // one code path for both role lanes
                const bool t = lane == RT;
                const float *xs = t ? nullptr : (OCT < 8 ? csrc : role_src(enn, (int)__ldg(A.toct + vt + 1)));
                const float *ns = t ? A.vtab + (int64_t)(vt + 1) * kTabRows * kWarp : (xs ? xs + (vl + 1) * cstride : nullptr);
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
                acc[q] = ffma2(cdir[2], ld2(&F[q + NQ * lz][c2]), acc[q]);
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
                st2(&F[q + NQ * lz][c2 ^ (4 * (q & 7))], o);
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
                        lsum = ffma2(dup2(A.ops.wq[q % N1] * A.ops.wq[q / N1]), acc[q], lsum);
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
                using FP_ = std::integral_constant<bool, GEN == 2>;
                if (A.limiter)
                    A.vtau ? bgk_src(T_{}, FP_{}, T_{}) : bgk_src(F_{}, FP_{}, T_{});
                else
                    A.vtau ? bgk_src(T_{}, FP_{}, F_{}) : bgk_src(F_{}, FP_{}, F_{});
            } else {
                bgk_src(F_{}, F_{}, F_{});
            }
            if (GEN && A.limiter) {
                // Zhang-Shu (Sec. 2.1, Eqs. 10-11): element mean and minimum of every velocity over the
                // layers, then the contraction of the values of this half-warp's layer
                st2(&sm.lim[0][lz][c2], fmul2(dup2(A.ops.wq[lz]), lsum));
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
                const float *ys = OCT < 8 ? csrc : role_src(enn, (int)__ldg(A.toct + vt + 1));
                fence_proxy_async();
                issue(ys, vl + 1, bF);
            }
#pragma unroll
            for (int d = 0; d < 3; d++)
                en[d] = enn[d];
            const int t = bF;
            bF = bX;
            bX = bN;
            bN = bY;
            bY = t;
        }
        // the end of a moment group: combine the 4 velocity eighths of a row
        const int grp = moment_group(A, blockIdx.x / E, vl - 1);
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
}

template <int N1, int OCT, int GEN>
cudaError_t launch3s(const StageArgs &A0, cudaStream_t s)
{
    using Sm = Stage3sSmem<N1, GEN>;
    static_assert(offsetof(Sm, tab) % 16 == 0 && offsetof(Sm, par) % 16 == 0 && offsetof(Sm, fpar) % 16 == 0 &&
                      offsetof(Sm, lim) % 16 == 0 && offsetof(Sm, bar) % 8 == 0,
                  "8- and 16-byte shared accesses");
    StageArgs A = A0;
    plan_tasks(A, A.mesh.nelem, 152 * kStage3sCtas<GEN>, 0.8, 0.75);
    k_stage3s<N1, OCT, GEN><<<A.mesh.nelem * A.ntasks, kWarp * N1 / 2, sizeof(Sm), s>>>(A);
    return cudaGetLastError();
}

template <int N1>
cudaError_t prepare3s()
{
    const int s0 = (int)sizeof(Stage3sSmem<N1, 0>), s1 = (int)sizeof(Stage3sSmem<N1, 1>);
    const int s2 = (int)sizeof(Stage3sSmem<N1, 2>);
    cudaError_t e = cudaSuccess;
#define BGK_P3S(O)                                                                                       \
    if (e == cudaSuccess)                                                                                \
        e = cudaFuncSetAttribute(k_stage3s<N1, O, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, s0); \
    if (e == cudaSuccess)                                                                                \
        e = cudaFuncSetAttribute(k_stage3s<N1, O, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, s1); \
    if (e == cudaSuccess)                                                                                \
        e = cudaFuncSetAttribute(k_stage3s<N1, O, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, s2);
    BGK_P3S(0) BGK_P3S(1) BGK_P3S(2) BGK_P3S(3) BGK_P3S(4) BGK_P3S(5) BGK_P3S(6) BGK_P3S(7) BGK_P3S(8)
#undef BGK_P3S
    return e;
}

template <int N1, int GEN>
cudaError_t launch3s_oct(const StageArgs &A, int oct, cudaStream_t s)
{
    switch (oct) {
    case 0: return launch3s<N1, 0, GEN>(A, s);
    case 1: return launch3s<N1, 1, GEN>(A, s);
    case 2: return launch3s<N1, 2, GEN>(A, s);
    case 3: return launch3s<N1, 3, GEN>(A, s);
    case 4: return launch3s<N1, 4, GEN>(A, s);
    case 5: return launch3s<N1, 5, GEN>(A, s);
    case 6: return launch3s<N1, 6, GEN>(A, s);
    case 7: return launch3s<N1, 7, GEN>(A, s);
    default: return launch3s<N1, 8, GEN>(A, s);
    }
}

}  // namespace bgk
