// Two time steps per launch of the isotropic acoustic scheme (2-D), the temporal blocking
// of the probed sweeps.
//
// The probed method keeps no wavefield history, so between the two steps of a pair only
// what the probe contraction reads has to reach HBM: the forward increment d^{n+1} (the
// contraction forms u_tt from two increments) or, in the adjoint, v^{j} itself.  u^{n+1}
// stays on chip.  Per shot and point a pair moves 8 B in (u^n, d^n) and 12 B out
// (d^{n+1} or u^{n+1}, then u^{n+2}, d^{n+2}) instead of 32 B for two single steps.
//
// Each step is the arithmetic of stencil_kernel, operation for operation, so a pair gives
// the same bits as two single-step launches.
//
// Tiling.  A block owns TX columns (4 per thread, one float4) and a segment of tz2
// planes.  Stage A computes step 1 on the whole TX-column tile and on the segment
// extended by 4 planes on either side; stage B computes step 2 on the inner TX - 8
// columns (the core) and the segment itself.  Neighbouring tiles overlap by 8 columns and
// neighbouring segments by 8 planes of stage-A work: the halo of step 2 is recomputed
// rather than exchanged.  Stage B trails stage A by 4 planes: u^{n+1} of the own float4
// lives in a register window, its x neighbours in a shared ring of 8 planes, and d^{n+1}
// replaces d^n in the ring slot it came from.
//
// What bounds it: a plane of the march is one long chain of instructions per warp (12 warps a
// SM, all the registers and shared memory allow), so its time is the number of instructions
// times their latency, as long as the loop stays in the instruction cache.  Hence
//   - every shared-memory access has a constant offset from one of two registers (rings of two
//     groups of four planes) and every global one is one multiply-add away from one offset;
//   - nothing outside the grid is tested: staging zero-fills it, and dt^2/m = 0 there makes both
//     steps give zero; the absorbing layer is a branch of the whole warp;
//   - the constants stay in registers (stencil_step.cuh), and groups without injection entries
//     run a copy of the loop without the lookups;
//   - the loop is unrolled by four planes: 185 instructions a warp and plane in 13 KB.  By three
//     it needs ring arithmetic (374 instructions a plane, 18 KB); by eight it drops the moves of
//     the register windows but stalls on instruction fetch (27 KB: 270 us where four planes take
//     218 and three took 300).
// Measured per launch of the 1601 x 401 model (padded 1681 x 481): 64 shots 218 us (300 before;
// 4.75 TB/s of the 20 B per point and shot it must move), 32 shots 121 (167), 16 shots 68 (94.5),
// 8 shots 41 (57), one shot 13 (33); with the imaging condition, 16 shots: 116 us (150 before,
// 130 without the L2 prefetch).  Launches of few blocks run stencil2_tile_kernel (below): one shot
// of 201 x 201 4.5 us (39 before, 10.0 marching in 3-plane segments), of 401 x 401 5.9 (9.9).
//
// Injection uses a CSR table keyed by (tile, plane of the extended segment) that lists
// every entry inside the extended tile (points in an overlap appear in both tiles);
// stage B reads the same keys and keeps the entries of its core.  Each warp sums the
// entries of its own columns in shared memory, so injection needs no block barrier.
//
// Recording: the extra blocks record R u^n from the input and, when the previous launch
// was a pair, the row of its first step as R (u^{n-1} + d^n) from the input of that launch
// and the stored increment, the same addition stage A made.
#include <cstdlib>
#include <type_traits>

#include "stencil_step.cuh"

namespace wp {

using step::P4;
using step::f2;


template <int TXT>
struct Stencil2Shape {
    static constexpr int TX = 4 * TXT;
    static constexpr int C = TX - 2 * RAD;          // core columns (stage B)
    static constexpr int NT = TXT;
    static constexpr int W = TX + 2 * RAD;          // u ring row (x halos of stage A)
    static constexpr int U = 4;                     // planes per unrolled group
    static constexpr int NR = 8;                    // ring slots (two groups)
    static constexpr int LA = 3;                    // planes in flight
    static constexpr int SLOT = W + 3 * TX;         // u^n row with halos, increment, dt^2/m, u^{n+1}
    // (the last lane reads one float4 past the u^{n+1} ring)
    static constexpr size_t SMEM = ((size_t)NR * SLOT + 4) * sizeof(float);
    // 6 blocks of 64 threads (33 KB of rings each) or 12 of 32: registers <= 168
    static constexpr int MINB = 384 / NT;
    static_assert(NR == 2 * U && U == RAD && RAD + 1 + LA <= NR, "rings");
};

// IMG: the imaging condition of both steps at offset o of shot sh.
__device__ __forceinline__ void image_pair(const StencilArgs &A, long long sh, long long o, const P4 &v1, const P4 &un,
                                           const float *sdv)
{
    // exact imaging of both steps at an output float4, one image read and write
    // per launch: first u_tt of the first step (increments h2, h1) times its
    // output v1, then that of the second (h1, h0) times un,
    // each written as the one-step kernel writes its update, so a pair adds
    // bit for bit what two single steps add
    float v[4], v2[4];
    step::upk(v1.a, v[0], v[1]);
    step::upk(v1.b, v[2], v[3]);
    step::upk(un.a, v2[0], v2[1]);
    step::upk(un.b, v2[2], v2[3]);
    float4 *gi = (float4 *)(A.img + sh * A.img_ss + o);
    float4 gv4 = *gi;
    const long long p = sh * A.h_ss + o;
    const float4 h2 = *(const float4 *)(A.h2 + p), h1 = *(const float4 *)(A.h1 + p);
    const float4 h0 = *(const float4 *)(A.h0 + p);
    gv4.x += A.img_scale * ((1.f + sdv[0]) * h2.x - (1.f - sdv[0]) * h1.x) * v[0];
    gv4.y += A.img_scale * ((1.f + sdv[1]) * h2.y - (1.f - sdv[1]) * h1.y) * v[1];
    gv4.z += A.img_scale * ((1.f + sdv[2]) * h2.z - (1.f - sdv[2]) * h1.z) * v[2];
    gv4.w += A.img_scale * ((1.f + sdv[3]) * h2.w - (1.f - sdv[3]) * h1.w) * v[3];
    gv4.x += A.img_scale * ((1.f + sdv[0]) * h1.x - (1.f - sdv[0]) * h0.x) * v2[0];
    gv4.y += A.img_scale * ((1.f + sdv[1]) * h1.y - (1.f - sdv[1]) * h0.y) * v2[1];
    gv4.z += A.img_scale * ((1.f + sdv[2]) * h1.z - (1.f - sdv[2]) * h0.z) * v2[2];
    gv4.w += A.img_scale * ((1.f + sdv[3]) * h1.w - (1.f - sdv[3]) * h0.w) * v2[3];
    *gi = gv4;
}

template <int TXT, bool WD, bool IMG>
__global__ void __launch_bounds__(TXT, Stencil2Shape<TXT>::MINB) stencil2_kernel(const GridDev G, const StencilArgs A)
{
    using S = Stencil2Shape<TXT>;
    constexpr int TX = S::TX, C = S::C, W = S::W, NT = S::NT, LA = S::LA, NR = S::NR, U = S::U;
    constexpr uint32_t SL = S::SLOT * 4, OD = W * 4, OB = OD + TX * 4, OV = OB + TX * 4;   // slot bytes, offsets
    extern __shared__ float4 smem4[];
    __shared__ float sq[2][TX];   // injected terms [stage][column]
    __shared__ int inj_lo, inj_hi;
    __shared__ f2 coef[8];

    const int ntx = (G.NXp + C - 1) / C;
    const int ntiles = ntx * ((G.NZ + G.tz2 - 1) / G.tz2);
    pdl_trigger();
    pdl_wait();
    if ((int)blockIdx.x >= ntiles) {
        gather_rows(A, blockIdx.x - ntiles);
        return;
    }
    const int lx = threadIdx.x, tile = blockIdx.x;
    const long long sh = blockIdx.y;
    const int x0 = (tile % ntx) * C - RAD;
    const int z0 = (tile / ntx) * G.tz2, z1 = min(z0 + G.tz2, G.NZ);
    const int zs = z0 - RAD, nrel = z1 - z0 + 2 * RAD;   // stage-A planes zs .. zs + nrel - 1
    const int KP = G.tz2 + 2 * RAD;                      // table keys per tile
    const int NXp = G.NXp, NZ = G.NZ;
    const int xc = x0 + 4 * lx;
    const bool a_ok = xc >= 0 && xc < NXp;               // the float4 lies inside the field
    const float *u = A.u_in + sh * A.u_in_ss;

    // Staging: thread lx copies float4 lx of the u row (x0 - 4 + 4 lx; lanes 0 and 1 also the
    // two last ones) and its own float4 of the increment and of dt^2/m.  Everything outside
    // the grid is zero-filled, where dt^2/m = 0 makes both steps give zero: stage A needs no
    // test for columns or planes beyond the grid.
    const int xu = x0 - RAD + 4 * lx, xv = xu + TX;
    const int nu = xu >= 0 && xu < NXp ? 16 : 0, nv = xv < NXp ? 16 : 0, nd = a_ok ? 16 : 0;
    const int own = a_ok ? xc : 0;
    // (a copy of zero bytes reads nothing, but its address stays inside the array)
    const float *gu = u + (nu ? xu : 0), *gv = u + (nv ? xv : 0);
    const float *gd = A.d_in + sh * A.d_in_ss + own, *gb = A.b + own;
    const uint32_t sb = (uint32_t)__cvta_generic_to_shared(smem4) + 16u * lx;
    // Plane zs + r (zeros outside the grid and past the segment) into the slot at `o`; ko: the
    // plane's offset in floats.  The tests are uniform over the block.
    const int ulim = min(NZ, z1 + 2 * RAD), dlim = min(NZ, z1 + RAD);
    auto issue_u = [&](int r, int ko, uint32_t o) {
        if ((unsigned)(zs + r) < (unsigned)ulim) {
            cp_async16(o, gu + ko, nu);
            if (lx < 2) cp_async16(o + TX * 4, gv + ko, nv);
        } else {
            step::sts(o, step::zero());
            if (lx < 2) step::sts(o + TX * 4, step::zero());
        }
    };
    auto issue_db = [&](int r, int ko, uint32_t o) {
        if ((unsigned)(zs + r) < (unsigned)dlim) {
            cp_async16(o + OD, gd + ko, nd);
            cp_async16(o + OB, gb + ko, nd);
        } else {
            step::sts(o + OD, step::zero());
            step::sts(o + OB, step::zero());
        }
    };

    // group g < LA holds u plane 4 + g and increment plane g; group 0 also u planes 0 .. 3
#pragma unroll
    for (int r = 0; r < RAD; r++) issue_u(r, (zs + r) * NXp, sb + r * SL);
#pragma unroll
    for (int g = 0; g < LA; g++) {
        issue_u(RAD + g, (zs + RAD + g) * NXp, sb + (RAD + g) * SL);
        issue_db(g, (zs + g) * NXp, sb + g * SL);
        cp_async_commit();
    }

    const int *off = A.inj ? A.inj_off + sh * ((long long)ntiles * KP + 1) : nullptr;
    const long long key0 = (long long)tile * KP;
    const bool tile_inj = off && off[key0] < off[key0 + KP];
    if (lx == 0) {
        inj_lo = 1 << 30;
        inj_hi = -(1 << 30);
        step::coef_store(&coef, G);
    }
    __syncthreads();
    if (tile_inj)
        for (int t = lx; t < KP; t += NT)
            if (off[key0 + t] < off[key0 + t + 1]) {
                atomicMin(&inj_lo, t);
                atomicMax(&inj_hi, t);
            }
    const float *trA = tile_inj ? A.traces + sh * A.tr_ss + (long long)A.step * A.tr_ts : nullptr;
    const float *trB = tile_inj ? A.traces + sh * A.tr_ss + (long long)A.step2 * A.tr_ts : nullptr;

    const bool st_ok = a_ok && lx >= 1 && lx <= TXT - 2;   // core float4 inside the field: stores
    float sdx[4];
#pragma unroll
    for (int j = 0; j < 4; j++) sdx[j] = damp_term(xc + j, G.nx, G.nbl, G.hs0x, G.inv_nbl);
    // the whole warp outside the x absorbing layers (columns outside the grid do not matter)
    const bool warp_int =
        __all_sync(0xffffffffu, !a_ok || (sdx[0] == 0.f && sdx[1] == 0.f && sdx[2] == 0.f && sdx[3] == 0.f));
    const int ri0 = G.nbl - zs, ri1 = G.nbl + G.nz - zs;   // rel of the planes outside the z layers
    float *uo = A.u_out + sh * A.u_out_ss + own, *dout = A.d_out + sh * A.d_out_ss + own;
    float *u1o = IMG ? nullptr : A.u1_out + sh * A.u1_ss + own;

    // Register windows of the own float4, slid by U planes after every group (first plane r0):
    // wa[i]: u^n of plane zs + r0 - 4 + i; wb[i]: u^{n+1} of plane zs + r0 - 8 + i.
    P4 wa[2 * RAD + U], wb[2 * RAD + U];
#pragma unroll
    for (int k = 0; k < RAD; k++) {
        const int zz = zs - RAD + k;
        wa[k] = (a_ok && zz >= 0) ? *(const P4 *)(u + (long long)zz * NXp + own) : step::zero();
    }
#pragma unroll
    for (int k = 0; k < 2 * RAD; k++) wb[k] = step::zero();
    cp_async_wait<LA - 1>();
    __syncthreads();
    const int klo = inj_lo, khi = inj_hi;
    const step::Coef K = step::coef_load(&coef);
#pragma unroll
    for (int k = 0; k < RAD; k++) wa[RAD + k] = step::lds(sb + 16 + (uint32_t)k * SL);

    // Plane r of the segment lies in slot r mod 8.  Groups of four planes start at slot 0 or 4:
    // slot s of the first kind is at s0 + s SL (s < 4) or s1 + s SL (s >= 4), s0 = s1 = sb in
    // even groups, s0 = sb + 4 SL and s1 = sb - 4 SL in odd ones, so every shared-memory access
    // has a constant offset from one of two registers.
    uint32_t s0 = sb, s1 = sb;
    // From here every array is addressed by the offset kz of plane rel - 4 (stage B's), one
    // multiply-add per access: the bases absorb the distance of the plane each one touches.
    int kz = (zs - RAD) * NXp;
    gu += (2 * RAD + LA) * (long long)NXp;
    gv += (2 * RAD + LA) * (long long)NXp;
    gd += (RAD + LA) * (long long)NXp;
    gb += (RAD + LA) * (long long)NXp;
    if (!IMG) u1o += RAD * (long long)NXp;
    const int warp = lx >> 5, lane = lx & 31;
    // Plane rel = group start + PH of stage A and, if doB (uniform), plane rel - 4 of stage B.
    // INJ: a source or receiver may lie in one of the two planes.
    auto plane = [&](auto phc, auto injc, int rel, bool doB) {
        constexpr int PH = decltype(phc)::value;
        constexpr bool INJ = decltype(injc)::value;
        auto slot = [&](auto sc) -> uint32_t {
            constexpr int q = decltype(sc)::value & (NR - 1);
            return (q < U ? s0 : s1) + q * SL;
        };
        const uint32_t qa = slot(std::integral_constant<int, PH>{});         // plane rel
        const uint32_t qb = slot(std::integral_constant<int, PH + RAD>{});   // planes rel - 4, rel + 4
        cp_async_wait<LA - 1>();
        __syncthreads();
        issue_u(rel + RAD + LA, kz, slot(std::integral_constant<int, PH + RAD + LA>{}));
        issue_db(rel + LA, kz, slot(std::integral_constant<int, PH + LA>{}));
        cp_async_commit();

        bool injA = false, injB = false;
        if (INJ) {
            int ea0 = 0, ea1 = 0, eb0 = 0, eb1 = 0;
            const int z = zs + rel;
            if (rel >= klo && rel <= khi && z >= 0 && z < NZ) {
                ea0 = off[key0 + rel];
                ea1 = off[key0 + rel + 1];
            }
            if (doB && rel - RAD >= klo && rel - RAD <= khi) {
                eb0 = off[key0 + rel - RAD];
                eb1 = off[key0 + rel - RAD + 1];
            }
            injA = ea1 > ea0;
            injB = eb1 > eb0;
            if (injA || injB) {
                // each warp sums the entries of its own 128 columns (no block barrier: a
                // lane only reads the float4 of its own columns after the warp's sync)
                *(float4 *)&sq[0][4 * lx] = make_float4(0.f, 0.f, 0.f, 0.f);
                *(float4 *)&sq[1][4 * lx] = make_float4(0.f, 0.f, 0.f, 0.f);
                __syncwarp();
                for (int e = ea0 + lane; e < ea1; e += 32) {
                    const InjEntry E = A.inj[e];
                    if ((E.a >> 7) == warp)
                        atomicAdd(&sq[0][E.a], E.w * A.tr_sign * trA[(long long)E.trace * A.tr_rs]);
                }
                for (int e = eb0 + lane; e < eb1; e += 32) {
                    const InjEntry E = A.inj[e];
                    if ((E.a >> 7) == warp && E.a >= RAD && E.a < TX - RAD)
                        atomicAdd(&sq[1][E.a], E.w * A.tr_sign * trB[(long long)E.trace * A.tr_rs]);
                }
                __syncwarp();
            }
        }

        if (IMG && st_ok && rel >= 2 * RAD - 2 && rel + 2 < nrel) {
            // stage B's history rows and image two planes ahead: into L2 (there are no registers
            // or shared memory left to bring them closer)
            const long long p = sh * A.h_ss + kz + own + 2 * (long long)NXp;
            prefetch_l2(A.h2 + p);
            prefetch_l2(A.h1 + p);
            prefetch_l2(A.h0 + p);
            prefetch_l2(A.img + sh * A.img_ss + kz + own + 2 * (long long)NXp);
        }
        const P4 bl = step::lds(qb + OV - 16), br = step::lds(qb + OV + 16);   // x neighbours of stage B

        // ---- stage A: step 1 at plane rel on the whole tile
        wa[2 * RAD + PH] = step::lds(qb + 16);
        const P4 al = step::lds(qa), ar = step::lds(qa + 32);
        const P4 adin = step::lds(qa + OD), ab = step::lds(qa + OB);
        P4 u1, d1;
        float sdv[4];
        step::step4<false, WD>(&wa[PH], nullptr, nullptr, al, ar, adin, ab, &sq[0][4 * lx], injA,
                               warp_int && rel >= ri0 && rel < ri1, sdx, zs + rel, G, K, d1, u1, sdv);
        step::sts(qa + OD, d1);   // d^{n+1} replaces d^n: stage B reads it 4 planes later
        step::sts(qa + OV, u1);
        wb[2 * RAD + PH] = u1;
        if (!IMG && st_ok && rel >= RAD && rel < nrel - RAD) *(P4 *)(u1o + kz) = u1;

        // ---- stage B: step 2 at plane rel - 4 on the core
        if (doB) {
            const P4 bdin = step::lds(qb + OD), bb = step::lds(qb + OB);
            const P4 v1 = wb[PH + RAD];
            P4 un, dn;
            step::step4<false, WD>(&wb[PH], nullptr, nullptr, bl, br, bdin, bb, &sq[1][4 * lx], injB,
                                   warp_int && rel - RAD >= ri0 && rel - RAD < ri1, sdx, zs + rel - RAD, G, K, dn, un,
                                   sdv);
            if (st_ok) {
                *(P4 *)(uo + kz) = un;
                *(P4 *)(dout + kz) = dn;
                if (IMG) {
                    image_pair(A, sh, kz + own, v1, un, sdv);
                }
            }
        }
        kz += NXp;
    };
    auto group = [&](auto injc, int r0) {
        const bool doB = r0 >= NR;   // stage B starts four planes after stage A's first core plane
        plane(std::integral_constant<int, 0>{}, injc, r0, doB);
        if (r0 + 1 < nrel) plane(std::integral_constant<int, 1>{}, injc, r0 + 1, doB);
        if (r0 + 2 < nrel) plane(std::integral_constant<int, 2>{}, injc, r0 + 2, doB);
        if (r0 + 3 < nrel) plane(std::integral_constant<int, 3>{}, injc, r0 + 3, doB);
    };
    uint32_t flip = U * SL;
    for (int r0 = 0; r0 < nrel; r0 += U) {
        // groups without injection entries (all but a few) run without the lookups
        if (klo < r0 + U && khi >= r0 - RAD) group(std::true_type{}, r0);
        else group(std::false_type{}, r0);
#pragma unroll
        for (int k = 0; k < 2 * RAD; k++) {
            wa[k] = wa[k + U];
            wb[k] = wb[k + U];
        }
        s0 += flip;
        s1 -= flip;
        flip = 0u - flip;
    }
    cp_async_wait<0>();
}

// Two steps of a small launch.  Marching fills a ring, then walks segment + 8 planes one after the
// other; where the chip has room for the whole launch at once, the planes of a segment can run side
// by side instead: a block holds all u^n rows of its tile in shared memory, every warp computes
// step 1 of its plane (two planes at 256 columns) and, after one barrier, step 2.  Same tiles, same
// keys of the injection tables and the same arithmetic as the march, so the same bits.
// Segments have at most MAXZ planes: 16 extended planes a block (twice the segment's work in step 1,
// in the time of one plane).  What bounds it: one latency of the L2 cache, the two steps' chains of
// instructions and the launch; a block of 512 threads takes an SM, and further rounds of blocks cost
// 2.7 us each, which is where the march overtakes it (choose_tz2).
template <int TXT>
struct Stencil2Tile {
    static constexpr int TX = 4 * TXT, C = TX - 2 * RAD, W = TX + 2 * RAD;
    static constexpr int NT = 512, PAR = NT / TXT;              // threads; planes side by side
    static constexpr int MAXZ = STENCIL2_TILE_Z, PL = MAXZ + 2 * RAD, NP = PL / PAR;   // planes a thread
    static constexpr int UR = PL + 2 * RAD;                     // u^n rows
    static constexpr size_t SMEM = ((size_t)(UR + PL) * W + NT * 4) * sizeof(float);
    static_assert(PL % PAR == 0, "planes");
};

template <int TXT, bool WD, bool IMG>
__global__ void __launch_bounds__(512, 1) stencil2_tile_kernel(const GridDev G, const StencilArgs A)
{
    using S = Stencil2Tile<TXT>;
    constexpr int C = S::C, W = S::W, NP = S::NP, PAR = S::PAR, TX = S::TX;
    extern __shared__ float4 smem4[];
    __shared__ f2 coef[8];
    const int ntx = (G.NXp + C - 1) / C;
    const int ntiles = ntx * ((G.NZ + G.tz2 - 1) / G.tz2);
    if (threadIdx.x == 0) step::coef_store(&coef, G);
    pdl_trigger();
    pdl_wait();
    if ((int)blockIdx.x >= ntiles) {
        gather_rows(A, blockIdx.x - ntiles);
        return;
    }
    const int lx = threadIdx.x % TXT, py = threadIdx.x / TXT, tile = blockIdx.x;
    const long long sh = blockIdx.y;
    const int x0 = (tile % ntx) * C - RAD;
    const int z0 = (tile / ntx) * G.tz2, z1 = min(z0 + G.tz2, G.NZ);
    const int zs = z0 - RAD, nrel = z1 - z0 + 2 * RAD;   // stage-A planes zs .. zs + nrel - 1
    const int KP = G.tz2 + 2 * RAD;
    const int NXp = G.NXp, NZ = G.NZ, xc = x0 + 4 * lx;
    const bool a_ok = xc >= 0 && xc < NXp;
    const float *u = A.u_in + sh * A.u_in_ss;
    const uint32_t su = (uint32_t)__cvta_generic_to_shared(smem4), sv = su + S::UR * W * 4;   // u^n and u^{n+1} rows
    // u^n rows of planes zs - 4 .. z1 + 7, columns x0 - 4 ..: zeros outside the grid
    for (int c = threadIdx.x; c < (nrel + 2 * RAD) * (W / 4); c += S::NT) {
        const int row = c / (W / 4), k = c - row * (W / 4);
        const int x = x0 - RAD + 4 * k, z = zs - RAD + row;
        const bool in = x >= 0 && x < NXp && z >= 0 && z < NZ;
        cp_async16(su + 16u * c, u + (in ? z * NXp + x : 0), in ? 16 : 0);
    }
    cp_async_commit();
    // own increment and dt^2/m (zeros outside the grid, where both steps then give zero)
    P4 d[NP], b[NP];
    const int *off = A.inj ? A.inj_off + sh * ((long long)ntiles * KP + 1) + (long long)tile * KP : nullptr;
    int e0[NP], e1[NP];
#pragma unroll
    for (int i = 0; i < NP; i++) {
        const int r = py + i * PAR, z = zs + r;
        const bool in = r < nrel && z >= 0 && z < NZ;
        d[i] = b[i] = step::zero();
        e0[i] = e1[i] = 0;
        if (in && a_ok) {
            d[i] = *(const P4 *)(A.d_in + sh * A.d_in_ss + z * NXp + xc);
            b[i] = *(const P4 *)(A.b + z * NXp + xc);
        }
        if (in && off) {
            e0[i] = off[r];
            e1[i] = off[r + 1];
        }
    }
    const float *trA = A.inj ? A.traces + sh * A.tr_ss + (long long)A.step * A.tr_ts : nullptr;
    const float *trB = A.inj ? A.traces + sh * A.tr_ss + (long long)A.step2 * A.tr_ts : nullptr;
    const bool st_ok = a_ok && lx >= 1 && lx <= TXT - 2;
    float sdx[4];
#pragma unroll
    for (int j = 0; j < 4; j++) sdx[j] = damp_term(xc + j, G.nx, G.nbl, G.hs0x, G.inv_nbl);
    const bool warp_int =
        __all_sync(0xffffffffu, !a_ok || (sdx[0] == 0.f && sdx[1] == 0.f && sdx[2] == 0.f && sdx[3] == 0.f));
    const int ri0 = G.nbl - zs, ri1 = G.nbl + G.nz - zs;
    const int lane = threadIdx.x & 31, half = lx >> 5;   // the warp's 128 columns of the tile
    float *sq = (float *)smem4 + (S::UR + S::PL) * W + (threadIdx.x - lane) * 4;   // injected terms of them
    // the terms of entries [a, e) in the warp's columns at or after lo and before hi
    auto inject = [&](int a, int e, const float *tr, int lo, int hi) {
        if (a >= e) return false;
        __syncwarp();
        *(float4 *)&sq[4 * lane] = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncwarp();
        for (int t = a + lane; t < e; t += 32) {
            const InjEntry E = A.inj[t];
            if ((E.a >> 7) == half && E.a >= lo && E.a < hi)
                atomicAdd(&sq[E.a & 127], E.w * A.tr_sign * tr[(long long)E.trace * A.tr_rs]);
        }
        __syncwarp();
        return true;
    };
    cp_async_wait<0>();
    __syncthreads();
    const step::Coef K = step::coef_load(&coef);
    const uint32_t ou = su + 16u * lx, ov = sv + 16u * lx;
    // ---- stage A: step 1 at every plane of the extended segment
    P4 u1[NP];
#pragma unroll
    for (int i = 0; i < NP; i++) {
        const int r = py + i * PAR;
        if (r >= nrel) break;
        const bool inj = inject(e0[i], e1[i], trA, 0, TX);
        P4 w[2 * RAD + 1], dn;
#pragma unroll
        for (int k = 0; k <= 2 * RAD; k++) w[k] = step::lds(ou + (uint32_t)(r + k) * (W * 4) + 16);
        const P4 al = step::lds(ou + (uint32_t)(r + RAD) * (W * 4)), ar = step::lds(ou + (uint32_t)(r + RAD) * (W * 4) + 32);
        float sdv[4];
        step::step4<false, WD>(w, nullptr, nullptr, al, ar, d[i], b[i], &sq[4 * lane], inj,
                               warp_int && r >= ri0 && r < ri1, sdx, zs + r, G, K, dn, u1[i], sdv);
        d[i] = dn;
        step::sts(ov + (uint32_t)r * (W * 4) + 16, u1[i]);
        if (!IMG && st_ok && r >= RAD && r < nrel - RAD)
            *(P4 *)(A.u1_out + sh * A.u1_ss + (zs + r) * NXp + xc) = u1[i];
    }
    __syncthreads();
    // ---- stage B: step 2 at the segment's own planes, on the core
#pragma unroll
    for (int i = 0; i < NP; i++) {
        const int r = py + i * PAR;
        if (r < RAD || r >= nrel - RAD) continue;
        const bool inj = inject(e0[i], e1[i], trB, RAD, TX - RAD);
        P4 w[2 * RAD + 1], dn, un;
#pragma unroll
        for (int k = 0; k <= 2 * RAD; k++) w[k] = step::lds(ov + (uint32_t)(r - RAD + k) * (W * 4) + 16);
        const P4 bl = step::lds(ov + (uint32_t)r * (W * 4)), br = step::lds(ov + (uint32_t)r * (W * 4) + 32);
        float sdv[4];
        step::step4<false, WD>(w, nullptr, nullptr, bl, br, d[i], b[i], &sq[4 * lane], inj,
                               warp_int && r >= ri0 && r < ri1, sdx, zs + r, G, K, dn, un, sdv);
        if (st_ok) {
            const int o = (zs + r) * NXp + xc;
            *(P4 *)(A.u_out + sh * A.u_out_ss + o) = un;
            *(P4 *)(A.d_out + sh * A.d_out_ss + o) = dn;
            if (IMG) image_pair(A, sh, o, u1[i], un, sdv);
        }
    }
}

template <int TXT, bool WD, bool IMG = false>
static void launch2_variant(const GridDev &G, const StencilArgs &A, dim3 grid, cudaStream_t s)
{
    if (G.side2) {
        using S = Stencil2Tile<TXT>;
        const dim3 tgrid(stencil2_tiles(G) + gather_blocks(A, S::NT), A.nshots);
        cudaFuncSetAttribute(stencil2_tile_kernel<TXT, WD, IMG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM);
        pdl_launch(stencil2_tile_kernel<TXT, WD, IMG>, tgrid, S::NT, S::SMEM, s, G, A);
        return;
    }
    using S = Stencil2Shape<TXT>;
    cudaFuncSetAttribute(stencil2_kernel<TXT, WD, IMG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM);
    pdl_launch(stencil2_kernel<TXT, WD, IMG>, grid, S::NT, S::SMEM, s, G, A);
}

template <int TXT>
static void launch2_tiles(const GridDev &G, const StencilArgs &A, cudaStream_t s)
{
    using S = Stencil2Shape<TXT>;
    dim3 grid(stencil2_tiles(G) + gather_blocks(A, S::NT), A.nshots);
    if (A.img) launch2_variant<TXT, false, true>(G, A, grid, s);   // exact adjoint: (u, d) form
    else if (A.wd) launch2_variant<TXT, true>(G, A, grid, s);
    else launch2_variant<TXT, false>(G, A, grid, s);
}

template <int TXT>
static int blocks2_per_sm()
{
    using S = Stencil2Shape<TXT>;
    static int cached = 0;
    if (!cached) {
        cudaFuncSetAttribute(stencil2_kernel<TXT, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM);
        int n = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, stencil2_kernel<TXT, true, false>, S::NT, S::SMEM) != cudaSuccess || n < 1)
            n = 1;
        cached = n;
    }
    return cached;
}

int stencil2_blocks_per_sm(const GridDev &G) { return G.tx == 128 ? blocks2_per_sm<32>() : blocks2_per_sm<64>(); }

cudaError_t launch_stencil2(const GridDev &G, const StencilArgs &A, cudaStream_t s)
{
    if (G.ndim != 2 || G.tti || G.tz2 < 1 || (G.tx != 128 && G.tx != 256)) return cudaErrorInvalidValue;
    if (G.side2 && G.tz2 > STENCIL2_TILE_Z) return cudaErrorInvalidValue;
    if (A.img && A.wd) return cudaErrorInvalidValue;   // the imaging pair is the adjoint's (u, d) form
    const int cls = A.img ? PROF_STENCIL2_IMG : PROF_STENCIL2;
    cudaEvent_t ev = prof_begin(cls, s);
    if (G.tx == 128) launch2_tiles<32>(G, A, s);
    else launch2_tiles<64>(G, A, s);
    prof_end(cls, ev, s);
    count_launch();
    return cudaGetLastError();
}

}  // namespace wp
