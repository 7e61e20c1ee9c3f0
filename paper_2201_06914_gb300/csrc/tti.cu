// Pseudo-acoustic TTI time step (the paper's second physics, Sec. 3 "2007 BP TTI"; the
// paper gives no equations).  Two fields per shot, stored as two consecutive "virtual
// shots" (field p at 2s, field q at 2s+1):
//   m (p_tt + sigma p_t) = E H0 p + S Hz q + src,   m (q_tt + sigma q_t) = S H0 p + Hz q + src
// with E = 1 + 2 eps, S = sqrt(1 + 2 delta), Hz = -Dr^T Dr = sum_i D_i (a_i Dr .),
// Dr = sum_i a_i D_i (8th-order central first derivatives, a = tilted symmetry axis) and
// H0 = L - Hz.  The adjoint applies the transposed block operator: it first combines
// e = E a + S b, f = S a + b and then applies H0 to e and Hz to f.  The adjoint step that
// updates (a, b) also writes the (e, f) of the new fields, so the next step reads them
// directly.
//
// One step = pass 1 (t_j = Dr x_j for both fields), pass 2 (Hz, L, combination and the
// increment-form leapfrog update of both fields, optionally the exact imaging condition
// summed over both fields), then a point-list injection that adds the linear source term
// to the updated increments and fields.  Both passes are tiled z-marching kernels in 3-D; in 2-D
// pass 1 and, on small launches, pass 2 read their neighbourhoods directly.
//
// What bounds them: 3-D pass 1 shared-memory reads, pass 2 instruction latency at 16 warps a SM and
// then DRAM (28 and 64 B a point); small 2-D launches one latency of the L2 cache per kernel.
// Measured (adjoint, padded 240 x 240 x 192): pass 1 74 us (232 instructions per field and 128
// points; 85 us and 368 for both fields in one thread, 93 us and 582 with two points a thread),
// pass 2 157 us, 478 per 64 points (201 us, 661: constants re-created at every use, IEEE divisions
// in a divergent branch, twelve copies a plane issued by one thread).  One step of the padded
// 336 x 336 x 272 grid: 571 us (737 before), of one shot of 401 x 401 in 2-D: 8.9 us (57).
#include <cuda.h>

#include <algorithm>
#include <cstring>

#include "plane_ring.cuh"
#include "stencil_step.cuh"

namespace wp {

namespace {

constexpr float D1C1 = 4.0f / 5.0f, D1C2 = -1.0f / 5.0f, D1C3 = 4.0f / 105.0f,
                D1C4 = -1.0f / 280.0f;

struct Pt {
    int x, y, z;
};

__device__ __forceinline__ Pt coords(const GridDev &G, long long p)
{
    const long long row = p / G.NXp;
    Pt c;
    c.x = (int)(p - row * G.NXp);
    c.z = (int)(row / G.NY);
    c.y = (int)(row - (long long)c.z * G.NY);
    return c;
}

}  // namespace

// Both passes march a tile of (x, y) points along z (grid: blockIdx.x = (x tile, y tile,
// z segment), blockIdx.y = shot); the in-plane neighbours of a plane come from shared-memory
// tiles with halos of 4 (zero outside the grid), the 9-plane z neighbourhood of a thread's
// own points from registers.

// 8-byte shared-memory load, and constants that stay in registers (a packed instruction takes a
// constant only from a register pair; the compiler would re-create it with two moves per use).
__device__ __forceinline__ step::f2 lds2(uint32_t addr)
{
    step::f2 v;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(addr));
    return v;
}

__device__ __forceinline__ void tma3(uint32_t dst, const CUtensorMap *map, int x, int y, int z, uint64_t *bar)
{
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
                 "[%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
                 "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void tma4(uint32_t dst, const CUtensorMap *map, int x, int y, int z, int w, uint64_t *bar)
{
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
                 "[%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
                 "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(bar))
                 : "memory");
}

// fetches a tensor map ahead of its first use (a kernel parameter: before the predecessor has ended)
__device__ __forceinline__ void tma_prefetch(const CUtensorMap *map)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

// Differences or sums of the x neighbours +k and -k of pair p (points x + 2p, x + 2p + 1) from
// the values f[x - 4 ..] held as aligned pairs q: even offsets are aligned pairs, odd ones two
// scalar operations (no re-pairing moves).
template <bool SUM>
__device__ __forceinline__ step::f2 xpm(const step::f2 *q, int k, int p = 0)
{
    const int i = 2 + p;
    if ((k & 1) == 0) return SUM ? step::add2(q[i + k / 2], q[i - k / 2]) : step::sub2(q[i + k / 2], q[i - k / 2]);
    auto v = [&](int j) {
        float lo, hi;
        step::upk(q[j >> 1], lo, hi);
        return (j & 1) ? hi : lo;
    };
    const int j = 2 * i;
    return SUM ? step::pk(__fadd_rn(v(j + k), v(j - k)), __fadd_rn(v(j + 1 + k), v(j + 1 - k)))
               : step::pk(__fsub_rn(v(j + k), v(j - k)), __fsub_rn(v(j + 1 + k), v(j + 1 - k)));
}

// Pass 1: t_j = Dr x_j = sum_i a_i D_i x_j for both fields; x_j are the fields (forward) or
// the combinations e = E a + S b, f = S a + b (adjoint).
//
// In 3-D it marches along z.  Half of a block's threads compute field 0 and half field 1: a thread
// with both holds two z windows (168 registers, 12 warps a SM) and waits half of its time; split,
// 24 warps take 74 instead of 85 us on a padded 240 x 240 x 192 grid, where the 28 B a point take
// 46 and the L1 cache's data path is 70 % busy.  Every thread owns two pairs of adjacent points of
// a row and works on pairs with the packed f32x2 instructions.  The x_j tiles of a plane (with x
// and y halos) and the a_x, a_y, a_z tiles of the block's own points are staged by two tiled TMA
// copies (zero fill outside the grid) into a ring of NS planes, LA planes ahead; a slot is refilled
// once every warp has read it, so warps may be a plane or two apart (a barrier per plane: 578
// instead of 571 us a step on 336 x 336 x 272).  The 9-plane z window of the own points is kept in
// registers, its newest plane loaded from global memory two iterations ahead.
template <int TXP, int TY>
struct Tti1Shape {
    static constexpr int H = 2;                      // pairs of points per thread
    static constexpr int TXT = TXP / (2 * H), NF = TXT * TY, NT = 2 * NF;   // threads per field and block
    static constexpr int WX = TXP + 2 * RAD, WY = TY + 2 * RAD;
    static constexpr int R32(int n) { return (n + 31) / 32 * 32; }   // 128-byte TMA destinations
    static constexpr int LA = 2, NS = 4, U = 2;      // planes in flight; ring slots; unrolled planes
    static constexpr int XT = WY * WX;               // floats of one field tile with halos
    static constexpr int AT = TY * TXP;              // floats of one own-point tile
    static constexpr int OA = R32(2 * XT), SLOT = OA + R32(3 * AT);   // x_0, x_1; a_x, a_y, a_z
    static constexpr uint32_t TX_BYTES = 4u * (2u * XT + 3u * AT);
    static constexpr size_t SMEM = (size_t)NS * SLOT * sizeof(float) + 128;
    static constexpr int MINB = 3;                   // 80 registers, 24 warps a SM
    static_assert(NF % 32 == 0, "fields by warp");
};

// Tensor maps of one pass-1 launch: x_0 and x_1 [virtual shot][z][y][x] in boxes of both fields,
// [a_x, a_y, a_z][z][y][x] in boxes of all three.
struct Tti1Maps {
    CUtensorMap x, a;
};

// two pairs from shared memory in one load
__device__ __forceinline__ void ldsp(uint32_t addr, step::f2 *v)
{
    const step::P4 q = step::lds(addr);
    v[0] = q.a;
    v[1] = q.b;
}

template <int TXP, int TY>
__global__ void __launch_bounds__(Tti1Shape<TXP, TY>::NT, Tti1Shape<TXP, TY>::MINB)
    tti_pass1_kernel(const GridDev G, const TtiArgs T, int tz, int ntx, int nty, const __grid_constant__ Tti1Maps M)
{
    using S = Tti1Shape<TXP, TY>;
    using step::f2;
    constexpr int TXT = S::TXT, H = S::H, NF = S::NF, WX = S::WX, XT = S::XT, AT = S::AT, LA = S::LA, NS = S::NS,
                  U = S::U;
    extern __shared__ float4 smem4[];
    __shared__ f2 coef[4];
    __shared__ uint64_t full[NS], empty[NS];
    const uint32_t ring = (smem_u32(smem4) + 127u) & ~127u;
    const int tid = threadIdx.x, f = tid / NF, tf = tid % NF, lx = tf % TXT, ly = tf / TXT;   // f: uniform in a warp
    const int bx = blockIdx.x % ntx, by = (blockIdx.x / ntx) % nty, seg = blockIdx.x / (ntx * nty);
    const int sh = blockIdx.y;
    const int x0 = bx * TXP, y0 = by * TY, z0 = seg * tz, z1 = min(z0 + tz, G.NZ);
    const int NXp = G.NXp, PS = G.NXp * G.NY;
    if (tid == 0) {
        tma_prefetch(&M.x);
        tma_prefetch(&M.a);
        for (int i = 0; i < NS; i++) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], S::NT / 32);
        }
        fence_mbar_init();
        const float cw[4] = {D1C1, D1C2, D1C3, D1C4};
#pragma unroll
        for (int k = 0; k < 4; k++) coef[k] = step::dup(cw[k]);
    }
    pdl_trigger();
    pdl_wait();
    __syncthreads();
    // the two copies of plane k into ring slot sl, issued by the first thread of either half
    auto issue = [&](int k, int sl) {
        if (tf != 0) return;
        const uint32_t b = ring + (uint32_t)sl * (S::SLOT * 4);
        if (f == 0) {
            mbar_arrive_expect_tx(&full[sl], S::TX_BYTES);
            tma4(b, &M.x, x0 - RAD, y0 - RAD, k, 2 * sh, &full[sl]);
        } else tma4(b + S::OA * 4, &M.a, x0, y0, k, 0, &full[sl]);
    };
    for (int g = 0; g < LA && z0 + g < z1; g++) issue(z0 + g, g);

    const int x = x0 + 2 * H * lx, y = y0 + ly;
    const bool row_ok = x < NXp && y < G.NY;      // the points lie in the (padded) row
    const int own = row_ok ? y * NXp + x : 0;
    const float *gf = (T.adjoint ? T.ef_in + (2LL * sh + f) * T.ef_ss : T.u_in + (2LL * sh + f) * T.u_in_ss) + own;
    // own points at offset o (`in`: uniform; zero outside the grid)
    auto ldw = [&](f2 *v, bool in, int o) {
#pragma unroll
        for (int p = 0; p < H; p++) v[p] = 0ull;
        if (!row_ok || !in) return;
        const step::P4 a = *(const step::P4 *)(gf + o);
        v[0] = a.a;
        v[1] = a.b;
    };
    f2 w[2 * RAD + U][H];   // w[ph + 4 + k]: plane zb + ph + k (group start zb)
#pragma unroll
    for (int k = 0; k < 2 * RAD; k++) {
        const int zz = z0 - RAD + k;
        ldw(w[k], zz >= 0 && zz < G.NZ, zz * PS);
    }
    // the newest window plane (z+4) and the one after it, loaded two iterations ahead
    f2 p0[H], n0[H];
    ldw(p0, z0 + RAD < G.NZ, (z0 + RAD) * PS);
    ldw(n0, z0 + RAD + 1 < G.NZ, (z0 + RAD + 1) * PS);
    float *to = T.t + (2LL * sh + f) * T.t_ss + own;
    const f2 ihx = step::dup(1.f / G.hx), ihy = step::dup(1.f / G.hy), ihz = step::dup(1.f / G.hz);
    const uint32_t ox = (f * XT + (ly + RAD) * WX + RAD + 2 * H * lx) * 4;   // own points in the field tile
    const uint32_t oa = (S::OA + ly * TXP + 2 * H * lx) * 4;                // and in an own-point tile
    f2 ck[4];
#pragma unroll
    for (int k = 0; k < 4; k++) ck[k] = lds2(smem_u32(&coef[k]));
    const bool pad = x + 2 * H > G.NX;   // the points hold row padding: t = 0 there
    PlaneRing<NS, LA> pr;
    auto raise = [&] { if (T.err) atomicExch(T.err, 1); };
    int sc = 0;                          // ring slot of plane z
    uint32_t parity = 0, slot = ring;
    int kz = z0 * PS;
    for (int zb = z0; zb < z1; zb += U) {
#pragma unroll
        for (int ph = 0; ph < U; ph++) {
            const int z = zb + ph;
            if (z >= z1) break;
            if (tf == 0) {
                // plane z + LA takes the slot of plane z - (NS - LA), once every warp is past that
                const int si = sc + LA >= NS ? sc + LA - NS : sc + LA;
                pr.refill(z - z0, z1 - z0,
                          [&] { return mbar_wait_bounded(&empty[si], parity ^ (sc + LA >= NS ? 0u : 1u)); }, raise,
                          [&] { issue(z + LA, si); });
            }
            __syncwarp();
#pragma unroll
            for (int p = 0; p < H; p++) {
                w[2 * RAD + ph][p] = p0[p];
                p0[p] = n0[p];
            }
            ldw(n0, z + RAD + 2 < G.NZ, kz + (RAD + 2) * PS);
            // a wait that gives up sets the error flag; the march goes on without waiting or issuing
            pr.await(z - z0, z1 - z0, [&] { return mbar_wait_bounded(&full[sc], parity); }, raise);
            const uint32_t fb = slot + ox;
            f2 q[4 + H];   // x neighbours x-4 .. as aligned pairs
#pragma unroll
            for (int i = 0; i < 4 + H; i += H) ldsp(fb + (i - 2) * 8, q + i);
            f2 dx[H], dy[H], dz[H], t[H];
#pragma unroll
            for (int k = 1; k <= RAD; k++) {
                f2 yp[H], ym[H];
                ldsp(fb + k * WX * 4, yp);
                ldsp(fb - k * WX * 4, ym);
#pragma unroll
                for (int p = 0; p < H; p++) {
                    auto acc = [&](f2 v, f2 &h) { h = k == 1 ? step::mul2(ck[0], v) : step::fma2(ck[k - 1], v, h); };
                    acc(xpm<false>(q, k, p), dx[p]);
                    acc(step::sub2(w[ph + RAD + k][p], w[ph + RAD - k][p]), dz[p]);
                    acc(step::sub2(yp[p], ym[p]), dy[p]);
                }
            }
            f2 ax[H], ay[H], az[H];
            ldsp(slot + oa, ax);
            ldsp(slot + oa + AT * 4, ay);
            ldsp(slot + oa + 2 * AT * 4, az);
#pragma unroll
            for (int p = 0; p < H; p++) {
                f2 acc = step::mul2(step::mul2(ax[p], dx[p]), ihx);
                acc = step::fma2(step::mul2(ay[p], dy[p]), ihy, acc);
                t[p] = step::fma2(step::mul2(az[p], dz[p]), ihz, acc);
            }
            if (pad) {
#pragma unroll
                for (int p = 0; p < H; p++) {
                    float a, b;
                    step::upk(t[p], a, b);
                    t[p] = step::pk(x + 2 * p < G.NX ? a : 0.f, x + 2 * p + 1 < G.NX ? b : 0.f);
                }
            }
            if (row_ok) *(step::P4 *)(to + kz) = step::P4{t[0], t[1]};
            kz += PS;
            __syncwarp();
            if ((tid & 31) == 0) mbar_arrive(&empty[sc]);   // the warp has read the slot
            sc++;
            slot += S::SLOT * 4;
            if (sc == NS) {
                sc = 0;
                slot = ring;
                parity ^= 1;
            }
        }
#pragma unroll
        for (int k = 0; k < 2 * RAD; k++)
#pragma unroll
            for (int p = 0; p < H; p++) w[k][p] = w[k + U][p];
    }
    if (__syncthreads_or(pr.issued) && tf == 0)
        pr.drain(z1 - z0, [&](int i, uint32_t ph) { (void)mbar_wait_bounded(&full[i], ph); });
    __syncthreads();
}

// Pass 1 in 2-D, without shared memory: a thread computes one pair of points of one field in ZP
// consecutive planes.  It issues every load it needs (the pairs of ZP + 8 planes, four more x
// neighbours and two axis pairs a plane) before the first use, so a block takes one latency of the
// L2 cache, where the fields of 2-D grids mostly lie; x neighbours come from the L1 cache.  A march
// with a ring to fill first is no faster on small grids and slower on large ones: 4 shots of 1601 x
// 401 55 us a step (60.6 marching; 57 with 2 planes a thread, 56.5 with 8).
template <int ZP>
__global__ void __launch_bounds__(128) tti_pass1_2d_kernel(const GridDev G, const TtiArgs T)
{
    using step::f2;
    const int np = G.NXp / 2, gid = blockIdx.x * 128 + threadIdx.x;
    const int seg = gid / np, x = 2 * (gid - seg * np), z0 = seg * ZP;
    const long long vs = 2LL * blockIdx.y + blockIdx.z;   // virtual shot
    const int NXp = G.NXp;
    pdl_trigger();
    pdl_wait();
    if (z0 >= G.NZ) return;
    const float *f = (T.adjoint ? T.ef_in + vs * T.ef_ss : T.u_in + vs * T.u_in_ss) + z0 * NXp + x;
    const float *pax = T.ax + z0 * NXp + x, *paz = T.az + z0 * NXp + x;
    f2 w[ZP + 2 * RAD], q[ZP][5], ax[ZP], az[ZP];   // z window, pairs x - 4 .. x + 5 of a plane
#pragma unroll
    for (int k = 0; k < ZP + 2 * RAD; k++) {
        const int zz = z0 - RAD + k;
        w[k] = zz >= 0 && zz < G.NZ ? *(const f2 *)(f + (k - RAD) * NXp) : 0ull;
    }
#pragma unroll
    for (int j = 0; j < ZP; j++) {
        const bool in = z0 + j < G.NZ;
#pragma unroll
        for (int i = 0; i < 5; i++) {
            const int xx = x + 2 * (i - 2);
            q[j][i] = i == 2 ? w[RAD + j] : in && xx >= 0 && xx < NXp ? *(const f2 *)(f + j * NXp + 2 * (i - 2)) : 0ull;
        }
        ax[j] = in ? *(const f2 *)(pax + j * NXp) : 0ull;
        az[j] = in ? *(const f2 *)(paz + j * NXp) : 0ull;
    }
    float *t = T.t + vs * T.t_ss + z0 * NXp + x;
    const f2 ihx = step::dup(1.f / G.hx), ihz = step::dup(1.f / G.hz);
    const float cw[4] = {D1C1, D1C2, D1C3, D1C4};
#pragma unroll
    for (int j = 0; j < ZP; j++) {
        if (z0 + j >= G.NZ) break;
        f2 dx, dz;
#pragma unroll
        for (int k = 1; k <= RAD; k++) {
            const f2 c = step::dup(cw[k - 1]), vx = xpm<false>(q[j], k), vz = step::sub2(w[j + RAD + k], w[j + RAD - k]);
            dx = k == 1 ? step::mul2(c, vx) : step::fma2(c, vx, dx);
            dz = k == 1 ? step::mul2(c, vz) : step::fma2(c, vz, dz);
        }
        f2 r = step::fma2(step::mul2(az[j], dz), ihz, step::mul2(step::mul2(ax[j], dx), ihx));
        if (x + 2 > G.NX) {   // row padding: t = 0 there
            float a, b;
            step::upk(r, a, b);
            r = step::pk(x < G.NX ? a : 0.f, x + 1 < G.NX ? b : 0.f);
        }
        *(f2 *)(t + j * NXp) = r;
    }
}

// Pass 2: Hz x_j = sum_i D_i (a_i t_j), L x_0, combination and the increment-form leapfrog
// update of both fields (optionally the exact imaging condition summed over both fields).
//
// Every thread owns two adjacent points of a row and works on pairs with the packed f32x2
// instructions (four would need 120 registers for the three windows).  Each plane is staged with
// seven tiled TMA copies (cp.async.bulk.tensor, zero fill outside the grid) into a ring of NS
// planes, LA planes ahead, completing on the slot's mbarrier: both t and x_0 with x and y halos,
// a_x with the x halo, a_y with the y halo, and the block's own points of E, S and dt^2/m, of both
// increments and of the fields.  The z neighbourhood of the own pair (a_z t_0, a_z t_1, x_0) is a
// register window whose newest plane is loaded one iteration ahead (and in 3-D fetched into L2
// three ahead: 3 % of a 3-D step; in 2-D the fields are in L2 already).
template <int TXP, int TY, bool ADJ>
struct Tti2Shape {
    static constexpr int TXT = TXP / 2, NT = TXT * TY;
    static constexpr int HY = TY > 1 ? RAD : 0;
    static constexpr int WX = TXP + 2 * RAD, WY = TY + 2 * HY;
    static constexpr int R32(int n) { return (n + 31) / 32 * 32; }   // 128-byte TMA destinations
    static constexpr int BH = WY * WX, XH = TY * WX, YH = TY > 1 ? WY * TXP : 0, OWN = TY * TXP;
    static constexpr int NU = ADJ ? 2 : 1;           // fields staged (forward: a is x_0's centre)
    static constexpr int OT = 0, OX0 = R32(2 * BH), OAX = OX0 + R32(BH), OAY = OAX + R32(XH), OPAR = OAY + R32(YH),
                         OD = OPAR + R32(3 * OWN), OU = OD + R32(2 * OWN), SLOT = OU + R32(NU * OWN);   // floats
    static constexpr int LA = 2, NS = 3, U = 2;
    static constexpr uint32_t TX_BYTES = 4u * (3u * BH + XH + YH + (3u + 2u + NU) * OWN);
    static constexpr size_t SMEM = (size_t)NS * SLOT * 4 + 128 + 64;
};

// Tensor maps of one pass-2 launch (encoded on the host per launch).
struct Tti2Maps {
    CUtensorMap t;      // [virtual shot][z][y][x] of t, box WX x WY of both fields
    CUtensorMap x0;     // x_0 field (a forward, e adjoint), box WX x WY
    CUtensorMap ax;     // [z][y][x], box WX x TY
    CUtensorMap ay;     // box TXP x WY
    CUtensorMap par;    // [E, S, dt^2/m][z][y][x], box TXP x TY of all three
    CUtensorMap d;      // increments [virtual shot][z][y][x], box TXP x TY of both fields
    CUtensorMap u;      // fields, box TXP x TY of both (adjoint) or of b alone (forward)
};

// absorbing-layer term of a pair of points along x (and y); the z term is added per plane
__device__ __forceinline__ step::f2 damp_xy2(const GridDev &G, int x, int y)
{
    const float sy = G.ndim == 3 ? damp_term(y, G.ny, G.nbl, G.hs0y, G.inv_nbl) : 0.f;
    return step::pk(damp_term(x, G.nx, G.nbl, G.hs0x, G.inv_nbl) + sy,
                    damp_term(x + 1, G.nx, G.nbl, G.hs0x, G.inv_nbl) + sy);
}

// The absorbing layer's factors of a pair of points: c = 1 + s, -c, 1 / c and 1 - s.
struct TtiLayer {
    step::f2 cp, ncp, rc, cm;
};
// Absorbing layer, s = sigma dt / 2: the update divides by 1 + s.  With rc the correctly
// rounded reciprocal of c = 1 + s, q = t rc corrected once by its exact remainder, q + (t -
// c q) rc, is the rounded quotient (Markstein 1990; 10^9 random t and c in 1 .. 3 gave the IEEE
// quotient each time) as long as the remainder does not underflow, and t itself where s = 0: three
// packed operations at every point instead of a branch around IEEE divisions.  For |t| below about
// 2^-107 (the foot of a wave front, 30 decades below the wave) the last bit can differ from the IEEE
// quotient, and an infinite t gives a NaN.  Those bits are enough to give the later rounding another
// draw: against the IEEE quotient the outputs of a 1000-step 2-D sweep differ by 6e-6, and the
// errors of either against 64 bits are the same (mean ratio 0.998 over 53 outputs of 27 cases, 2-D
// and 3-D).  Dividing in the layer gives the former bits and takes 94.3 instead of 84.7 ms on the
// adjoint of 256 x 256 x 192 and 11.8 instead of 9.4 on the forward of 401 x 401.
__device__ __forceinline__ TtiLayer tti_layer(const GridDev &G, step::f2 sdxy, int z)
{
    const step::f2 sd = step::add2(sdxy, step::dup(damp_term(z, G.nz, G.nbl, G.hs0z, G.inv_nbl)));
    TtiLayer L;
    float c0, c1;
    L.cp = step::add2(step::dup(1.f), sd);
    L.cm = step::sub2(step::dup(1.f), sd);
    step::upk(L.cp, c0, c1);
    L.ncp = step::pk(-c0, -c1);
    L.rc = step::pk(__frcp_rn(c0), __frcp_rn(c1));
    return L;
}

// What a step writes for shot sh, at the own points of plane 0.
struct TtiOut {
    float *u0, *u1, *d0, *d1, *e, *f;
};
template <bool ADJ>
__device__ __forceinline__ TtiOut tti_out(const TtiArgs &T, long long sh, int off)
{
    return {T.u_out + 2 * sh * T.u_out_ss + off, T.u_out + (2 * sh + 1) * T.u_out_ss + off,
            T.d_out + 2 * sh * T.d_out_ss + off, T.d_out + (2 * sh + 1) * T.d_out_ss + off,
            ADJ ? T.ef_out + 2 * sh * T.ef_ss + off : nullptr, ADJ ? T.ef_out + (2 * sh + 1) * T.ef_ss + off : nullptr};
}

// The end of a step for one pair of points, at offset k from the own points of plane 0 and p from
// the field's first: combination of L x_0, Hz x_0 and Hz x_1, the update of both increments and
// fields, the adjoint's new e and f and (IMG) the imaging condition.  pad: the pair holds row
// padding, which stays zero; own: its first point does not.
template <bool ADJ, bool IMG>
__device__ __forceinline__ void tti_update(const TtiArgs &T, const TtiOut &O, long long sh, int k, long long p, step::f2 lap,
                                           step::f2 H0, step::f2 H1, step::f2 cE, step::f2 cS, step::f2 cbm, step::f2 cd0,
                                           step::f2 cd1, step::f2 ca, step::f2 cbv, const TtiLayer &L, bool pad, bool own,
                                           bool row_ok)
{
    using step::f2;
    f2 r0, r1;
    if (!ADJ) {
        const f2 h0p = step::sub2(lap, H0);
        r0 = step::fma2(cE, h0p, step::mul2(cS, H1));
        r1 = step::fma2(cS, h0p, H1);
    } else {
        r0 = step::sub2(lap, H0);
        r1 = H1;
    }
    auto update = [&](f2 r, f2 dprev) {
        const f2 t = step::fma2(cbm, r, step::mul2(L.cm, dprev));
        const f2 q = step::mul2(t, L.rc);
        return step::fma2(step::fma2(L.ncp, q, t), L.rc, q);
    };
    f2 dn0 = update(r0, cd0), dn1 = update(r1, cd1);
    f2 un0 = step::add2(ca, dn0), un1 = step::add2(cbv, dn1);
    f2 e2 = 0ull, f2v = 0ull;
    if (ADJ) {
        e2 = step::fma2(cE, un0, step::mul2(cS, un1));
        f2v = step::fma2(cS, un0, un1);
    }
    if (pad) {
        auto padz = [&](f2 &v) {
            float lo, hi;
            step::upk(v, lo, hi);
            v = step::pk(own ? lo : 0.f, 0.f);
        };
        padz(un0);
        padz(un1);
        padz(dn0);
        padz(dn1);
        padz(e2);
        padz(f2v);
    }
    if (row_ok) {
        *(f2 *)(O.u0 + k) = un0;
        *(f2 *)(O.u1 + k) = un1;
        *(f2 *)(O.d0 + k) = dn0;
        *(f2 *)(O.d1 + k) = dn1;
        if (ADJ) {
            *(f2 *)(O.e + k) = e2;
            *(f2 *)(O.f + k) = f2v;
        }
        if (IMG) {
            const float *h1a = T.h1 + (2LL * sh) * T.h_ss, *h0a = T.h0 + (2LL * sh) * T.h_ss;
            const float *h1b = T.h1 + (2LL * sh + 1) * T.h_ss, *h0b = T.h0 + (2LL * sh + 1) * T.h_ss;
            const f2 ua = step::sub2(step::mul2(L.cp, *(const f2 *)(h1a + p)), step::mul2(L.cm, *(const f2 *)(h0a + p)));
            const f2 ub = step::sub2(step::mul2(L.cp, *(const f2 *)(h1b + p)), step::mul2(L.cm, *(const f2 *)(h0b + p)));
            f2 *gi = (f2 *)(T.img + (long long)sh * T.img_ss + p);
            const f2 add = step::mul2(step::dup(T.img_scale), step::fma2(ua, un0, step::mul2(ub, un1)));
            f2 g = step::add2(*gi, add);
            if (pad) {
                float lo, hi;
                step::upk(g, lo, hi);
                g = step::pk(own ? lo : 0.f, 0.f);
            }
            *gi = g;
        }
    }
}

// Pass 2 in 2-D on small launches, as tti_pass1_2d_kernel: one pair of points of both fields in ZP
// consecutive planes per thread, every load issued before the first use, no shared memory (168
// registers, 3 blocks a SM).  What bounds it is one latency of the L2 cache and the launch: a step
// of one shot of 401 x 401 takes 8.9 us, 11.8 with the marching kernel, which has a ring and its
// windows to fill for 3 planes a block (401 x 401 is one wave of this kernel).
template <int ZP, bool ADJ, bool IMG>
__global__ void __launch_bounds__(128) tti_pass2_2d_kernel(const GridDev G, const TtiArgs T)
{
    using step::f2;
    const int np = G.NXp / 2, gid = blockIdx.x * 128 + threadIdx.x;
    const int seg = gid / np, x = 2 * (gid - seg * np), z0 = seg * ZP, NXp = G.NXp;
    const long long sh = blockIdx.y;
    const f2 sdxy = damp_xy2(G, x, 0);
    pdl_trigger();
    pdl_wait();
    if (z0 >= G.NZ) return;
    const int o = z0 * NXp + x;
    const float *t0 = T.t + 2 * sh * T.t_ss + o, *t1 = t0 + T.t_ss;
    const float *ua = T.u_in + 2 * sh * T.u_in_ss + o, *ub = ua + T.u_in_ss;
    const float *xf = ADJ ? T.ef_in + 2 * sh * T.ef_ss + o : ua;
    const float *d0 = T.d_in + 2 * sh * T.d_in_ss + o, *d1 = d0 + T.d_in_ss;
    // z windows of a_z t_0, a_z t_1 and x_0; x neighbours of a_x t_0, a_x t_1 and x_0
    f2 wa[ZP + 2 * RAD], wb[ZP + 2 * RAD], wx[ZP + 2 * RAD], p0[ZP][5], p1[ZP][5], px[ZP][5];
    f2 E[ZP], S[ZP], b[ZP], da[ZP], db[ZP], va[ZP], vb[ZP];
    auto ld = [&](const float *f, int k) { return *(const f2 *)(f + k); };
#pragma unroll
    for (int k = 0; k < ZP + 2 * RAD; k++) {
        const int zz = z0 - RAD + k, r = (k - RAD) * NXp;
        const bool in = zz >= 0 && zz < G.NZ;
        const f2 az = in ? ld(T.az + o, r) : 0ull;
        wa[k] = step::mul2(az, in ? ld(t0, r) : 0ull);
        wb[k] = step::mul2(az, in ? ld(t1, r) : 0ull);
        wx[k] = in ? ld(xf, r) : 0ull;
    }
#pragma unroll
    for (int j = 0; j < ZP; j++) {
        const bool in = z0 + j < G.NZ;
        const int r = j * NXp;
#pragma unroll
        for (int i = 0; i < 5; i++) {
            const int xx = x + 2 * (i - 2), ri = r + 2 * (i - 2);
            const bool ok = in && xx >= 0 && xx < NXp;
            const f2 ax = ok ? ld(T.ax + o, ri) : 0ull;
            p0[j][i] = step::mul2(ax, ok ? ld(t0, ri) : 0ull);
            p1[j][i] = step::mul2(ax, ok ? ld(t1, ri) : 0ull);
            px[j][i] = i == 2 ? wx[RAD + j] : ok ? ld(xf, ri) : 0ull;
        }
        E[j] = in ? ld(T.E + o, r) : 0ull;
        S[j] = in ? ld(T.Sd + o, r) : 0ull;
        b[j] = in ? ld(T.b + o, r) : 0ull;
        da[j] = in ? ld(d0, r) : 0ull;
        db[j] = in ? ld(d1, r) : 0ull;
        va[j] = ADJ ? (in ? ld(ua, r) : 0ull) : wx[RAD + j];
        vb[j] = in ? ld(ub, r) : 0ull;
    }
    const TtiOut O = tti_out<ADJ>(T, sh, o);
    const f2 ihx = step::dup(1.f / G.hx), ihz = step::dup(1.f / G.hz), ihx2 = step::dup(G.ihx2), ihz2 = step::dup(G.ihz2);
    const float c1[4] = {D1C1, D1C2, D1C3, D1C4}, c2[4] = {WP_C1, WP_C2, WP_C3, WP_C4};
    const bool pad = x + 2 > G.NX, own = x < G.NX;
#pragma unroll
    for (int j = 0; j < ZP; j++) {
        if (z0 + j >= G.NZ) break;
        const f2 cc = step::add2(px[j][2], px[j][2]);
        f2 hx0, hx1, lxx, hz0, hz1, lzz;
#pragma unroll
        for (int k = 1; k <= RAD; k++) {
            const f2 cf = step::dup(c1[k - 1]), lf = step::dup(c2[k - 1]);
            auto acc = [&](f2 co, f2 v, f2 &h) { h = k == 1 ? step::mul2(co, v) : step::fma2(co, v, h); };
            acc(cf, xpm<false>(p0[j], k), hx0);
            acc(cf, xpm<false>(p1[j], k), hx1);
            acc(lf, step::sub2(xpm<true>(px[j], k), cc), lxx);
            acc(cf, step::sub2(wa[j + RAD + k], wa[j + RAD - k]), hz0);
            acc(cf, step::sub2(wb[j + RAD + k], wb[j + RAD - k]), hz1);
            acc(lf, step::sub2(step::add2(wx[j + RAD + k], wx[j + RAD - k]), cc), lzz);
        }
        const f2 H0 = step::fma2(hz0, ihz, step::mul2(hx0, ihx)), H1 = step::fma2(hz1, ihz, step::mul2(hx1, ihx));
        const f2 lap = step::fma2(lzz, ihz2, step::mul2(lxx, ihx2));
        tti_update<ADJ, IMG>(T, O, sh, j * NXp, o + j * NXp, lap, H0, H1, E[j], S[j], b[j], da[j], db[j], va[j], vb[j],
                               tti_layer(G, sdxy, z0 + j), pad, own, true);
    }
}

template <int TXP, int TY, bool ADJ, bool IMG>
__global__ void __launch_bounds__(Tti2Shape<TXP, TY, ADJ>::NT, TY > 1 ? 4 : 7)
    tti_pass2_kernel(const GridDev G, const TtiArgs T, int tz, int ntx, int nty, const __grid_constant__ Tti2Maps M)
{
    using S = Tti2Shape<TXP, TY, ADJ>;
    using step::f2;
    using step::pk;
    using step::upk;
    constexpr int TXT = S::TXT, HY = S::HY, WX = S::WX, LA = S::LA, NS = S::NS, U = S::U, OWN = S::OWN;
    extern __shared__ float4 smem4[];
    __shared__ f2 coef[8];
    __shared__ uint64_t full[NS];
    // 128-byte aligned by pointer arithmetic on the shared array (a shared pointer still)
    const uint32_t ring = (smem_u32(smem4) + 127u) & ~127u;
    const int tid = threadIdx.x, lx = tid % TXT, ly = tid / TXT, warp = tid >> 5, lane = tid & 31;
    const int bx = blockIdx.x % ntx, by = (blockIdx.x / ntx) % nty, seg = blockIdx.x / (ntx * nty);
    const int sh = blockIdx.y;
    const int x0 = bx * TXP, y0 = by * TY, z0 = seg * tz, z1 = min(z0 + tz, G.NZ);
    const int NXp = G.NXp, PS = G.NXp * G.NY;

    if (tid == 0) {
        tma_prefetch(&M.t);
        tma_prefetch(&M.x0);
        tma_prefetch(&M.ax);
        if (TY > 1) tma_prefetch(&M.ay);
        tma_prefetch(&M.par);
        tma_prefetch(&M.d);
        tma_prefetch(&M.u);
        for (int i = 0; i < NS; i++) mbar_init(&full[i], 1);
        fence_mbar_init();
        const float c8[8] = {D1C1, D1C2, D1C3, D1C4, WP_C1, WP_C2, WP_C3, WP_C4};
#pragma unroll
        for (int k = 0; k < 8; k++) coef[k] = step::dup(c8[k]);
    }
    pdl_trigger();
    pdl_wait();
    __syncthreads();
    // Producers: the seven copies of plane k into ring slot sl, shared between the warps' first
    // lanes (one thread issuing all of them held up its warp, and the block at the barrier).
    // The slot's phase completes once warp 0 has arrived and all bytes have landed.
    constexpr int NW = S::NT / 32;
    auto issue = [&](int k, int sl) {
        if (lane != 0) return;
        const uint32_t b = ring + (uint32_t)sl * (S::SLOT * 4);
        uint64_t *bar = &full[sl];
        if (warp == 0) {
            mbar_arrive_expect_tx(bar, S::TX_BYTES);
            tma4(b + S::OT * 4, &M.t, x0 - RAD, y0 - HY, k, 2 * sh, bar);
        }
        if (warp == 1 % NW) {
            tma4(b + S::OX0 * 4, &M.x0, x0 - RAD, y0 - HY, k, 2 * sh, bar);
            tma3(b + S::OAX * 4, &M.ax, x0 - RAD, y0, k, bar);
        }
        if (warp == 2 % NW) {
            if (TY > 1) tma3(b + S::OAY * 4, &M.ay, x0, y0 - HY, k, bar);
            tma4(b + S::OPAR * 4, &M.par, x0, y0, k, 0, bar);
        }
        if (warp == 3 % NW) {
            tma4(b + S::OD * 4, &M.d, x0, y0, k, 2 * sh, bar);
            tma4(b + S::OU * 4, &M.u, x0, y0, k, ADJ ? 2 * sh : 2 * sh + 1, bar);
        }
    };
    for (int g = 0; g < LA && z0 + g < z1; g++) issue(z0 + g, g);

    const int x = x0 + 2 * lx, y = y0 + ly;
    const bool row_ok = x < NXp && y < G.NY;
    const bool own = row_ok && x < G.NX;          // first point of the pair inside the row
    const int off = row_ok ? y * NXp + x : 0;
    const float *t0 = T.t + (2LL * sh) * T.t_ss + off;
    const float *t1 = T.t + (2LL * sh + 1) * T.t_ss + off;
    const float *xf = (ADJ ? T.ef_in + (2LL * sh) * T.ef_ss : T.u_in + (2LL * sh) * T.u_in_ss) + off;
    const float *azf = T.az + off;
    auto ld2 = [&](const float *f, int zz) -> f2 {
        return (row_ok && zz >= 0 && zz < G.NZ) ? *(const f2 *)(f + zz * PS) : 0ull;
    };
    // z windows: a_z t_0, a_z t_1, x_0 of plane zb + i - 4 at index i (group start zb)
    f2 wa[2 * RAD + U], wb[2 * RAD + U], wx[2 * RAD + U];
#pragma unroll
    for (int k = 0; k < 2 * RAD; k++) {
        const int zz = z0 - RAD + k;
        const f2 az = ld2(azf, zz);
        wa[k] = step::mul2(az, ld2(t0, zz));
        wb[k] = step::mul2(az, ld2(t1, zz));
        wx[k] = ld2(xf, zz);
    }
    f2 qa = ld2(azf, z0 + RAD), q0 = ld2(t0, z0 + RAD), q1 = ld2(t1, z0 + RAD), qx = ld2(xf, z0 + RAD);
    const TtiOut O = tti_out<ADJ>(T, sh, off);
    const f2 ihx = step::dup(1.f / G.hx), ihy = step::dup(1.f / G.hy), ihz = step::dup(1.f / G.hz);
    const f2 ihx2 = step::dup(G.ihx2), ihy2 = step::dup(G.ihy2), ihz2 = step::dup(G.ihz2);
    f2 cw[4], lw[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        cw[k] = lds2(smem_u32(&coef[k]));
        lw[k] = lds2(smem_u32(&coef[4 + k]));
    }
    const uint32_t ob = ((ly + HY) * WX + RAD + 2 * lx) * 4;   // own pair in a both-halo tile
    const uint32_t oxh = (ly * WX + RAD + 2 * lx) * 4;         // own pair in the a_x tile
    const uint32_t oyh = ((ly + HY) * TXP + 2 * lx) * 4;       // own pair in the a_y tile
    const uint32_t oo = (ly * TXP + 2 * lx) * 4;               // own pair in an own-point tile
    const f2 sdxy = damp_xy2(G, x, y);
    // the absorbing layer's factors change only in planes of the z layers
    TtiLayer L = tti_layer(G, sdxy, z0);
    const int zl0 = G.nbl, zl1 = G.nbl + G.nz;   // planes zl0 .. zl1 - 1 lie between the z layers
    const bool pad = x + 2 > G.NX;               // the pair holds row padding: kept at zero
    PlaneRing<NS, LA> pr;
    auto raise = [&] { if (T.err) atomicExch(T.err, 1); };
    int sc = 0;                                  // ring slot of plane z
    uint32_t parity = 0, slot = ring;
    int kz = z0 * PS;
    for (int zb = z0; zb < z1; zb += U) {
#pragma unroll
        for (int ph = 0; ph < U; ph++) {
            const int z = zb + ph;
            if (z >= z1) break;
            __syncthreads();   // slot of plane z-1 is free again
            pr.refill(z - z0, z1 - z0, [] { return true; }, raise,
                      [&] { issue(z + LA, sc + LA >= NS ? sc + LA - NS : sc + LA); });
            // own pair of plane z+4 enters the windows; plane z+5 is loaded
            wa[2 * RAD + ph] = step::mul2(qa, q0);
            wb[2 * RAD + ph] = step::mul2(qa, q1);
            wx[2 * RAD + ph] = qx;
            qa = q0 = q1 = qx = 0ull;
            if (row_ok && z + RAD + 1 < G.NZ) {
                const int k5 = kz + (RAD + 1) * PS;
                qa = *(const f2 *)(azf + k5);
                q0 = *(const f2 *)(t0 + k5);
                q1 = *(const f2 *)(t1 + k5);
                qx = *(const f2 *)(xf + k5);
            }
            if (TY > 1 && row_ok && z + RAD + 3 < G.NZ) {   // the window's planes two further, into L2
                const int k7 = kz + (RAD + 3) * PS;
                prefetch_l2(azf + k7);
                prefetch_l2(t0 + k7);
                prefetch_l2(t1 + k7);
                prefetch_l2(xf + k7);
            }
            if (z <= zl0 || z >= zl1) L = tti_layer(G, sdxy, z);
            // a wait that gives up sets the error flag; the march goes on without waiting or issuing
            pr.await(z - z0, z1 - z0, [&] { return mbar_wait_bounded(&full[sc], parity); }, raise);
            // x parts: five aligned pairs x-4 .. x+5 of t_0, t_1, x_0 and a_x
            f2 p0[5], p1[5], px[5];
#pragma unroll
            for (int i = 0; i < 5; i++) {
                const f2 a = lds2(slot + oxh + S::OAX * 4 + (i - 2) * 8);
                p0[i] = step::mul2(a, lds2(slot + ob + S::OT * 4 + (i - 2) * 8));
                p1[i] = step::mul2(a, lds2(slot + ob + (S::OT + S::BH) * 4 + (i - 2) * 8));
                px[i] = lds2(slot + ob + S::OX0 * 4 + (i - 2) * 8);
            }
            const f2 c = px[2], c2 = step::add2(c, c);
            f2 hx0, hx1, lxx, hy0 = 0ull, hy1 = 0ull, lyy = 0ull, hz0, hz1, lzz;
#pragma unroll
            for (int k = 1; k <= RAD; k++) {
                const f2 cf = cw[k - 1], lf = lw[k - 1];
                auto acc = [&](f2 co, f2 v, f2 &h) { h = k == 1 ? step::mul2(co, v) : step::fma2(co, v, h); };
                acc(cf, xpm<false>(p0, k), hx0);
                acc(cf, xpm<false>(p1, k), hx1);
                acc(lf, step::sub2(xpm<true>(px, k), c2), lxx);
                if (TY > 1) {
                    const f2 ap = lds2(slot + oyh + (S::OAY + k * TXP) * 4);
                    const f2 am = lds2(slot + oyh + (S::OAY - k * TXP) * 4);
                    const f2 y0p = step::mul2(ap, lds2(slot + ob + (S::OT + k * WX) * 4));
                    const f2 y0m = step::mul2(am, lds2(slot + ob + (S::OT - k * WX) * 4));
                    const f2 y1p = step::mul2(ap, lds2(slot + ob + (S::OT + S::BH + k * WX) * 4));
                    const f2 y1m = step::mul2(am, lds2(slot + ob + (S::OT + S::BH - k * WX) * 4));
                    acc(cf, step::sub2(y0p, y0m), hy0);
                    acc(cf, step::sub2(y1p, y1m), hy1);
                    const f2 xp = lds2(slot + ob + (S::OX0 + k * WX) * 4), xm = lds2(slot + ob + (S::OX0 - k * WX) * 4);
                    acc(lf, step::sub2(step::add2(xp, xm), c2), lyy);
                }
                acc(cf, step::sub2(wa[ph + RAD + k], wa[ph + RAD - k]), hz0);
                acc(cf, step::sub2(wb[ph + RAD + k], wb[ph + RAD - k]), hz1);
                acc(lf, step::sub2(step::add2(wx[ph + RAD + k], wx[ph + RAD - k]), c2), lzz);
            }
            f2 H0 = step::mul2(hx0, ihx), H1 = step::mul2(hx1, ihx), lap = step::mul2(lxx, ihx2);
            if (TY > 1) {
                H0 = step::fma2(hy0, ihy, H0);
                H1 = step::fma2(hy1, ihy, H1);
                lap = step::fma2(lyy, ihy2, lap);
            }
            H0 = step::fma2(hz0, ihz, H0);
            H1 = step::fma2(hz1, ihz, H1);
            lap = step::fma2(lzz, ihz2, lap);
            const uint32_t po = slot + oo;
            const f2 cE = lds2(po + S::OPAR * 4), cS = lds2(po + (S::OPAR + OWN) * 4);
            const f2 cbm = lds2(po + (S::OPAR + 2 * OWN) * 4);
            const f2 cd0 = lds2(po + S::OD * 4), cd1 = lds2(po + (S::OD + OWN) * 4);
            const f2 ca = ADJ ? lds2(po + S::OU * 4) : c, cbv = lds2(po + (S::OU + (ADJ ? OWN : 0)) * 4);
            tti_update<ADJ, IMG>(T, O, sh, kz, kz + off, lap, H0, H1, cE, cS, cbm, cd0, cd1, ca, cbv, L, pad, own, row_ok);
            kz += PS;
            sc++;
            slot += S::SLOT * 4;
            if (sc == NS) {
                sc = 0;
                slot = ring;
                parity ^= 1;
            }
        }
#pragma unroll
        for (int k = 0; k < 2 * RAD; k++) {
            wa[k] = wa[k + U];
            wb[k] = wb[k + U];
            wx[k] = wx[k + U];
        }
    }
    if (__syncthreads_or(pr.issued) && lane == 0)
        pr.drain(z1 - z0, [&](int i, uint32_t ph) { (void)mbar_wait_bounded(&full[i], ph); });
    __syncthreads();
}

// Adds the source term after the update: a point source value q at point p changes the
// increment and the field by (dt^2/m) q / (1 + sigma dt/2) (the update is linear in q).
// Forward: both fields; adjoint: the p-equation only.  The exact imaging condition gets
// the matching correction.
__global__ void tti_inject_kernel(const GridDev G, const TtiArgs T, const int *idx, const float *w,
                                  int npts, int ncorner, const float *traces, long long tr_ss,
                                  long long tr_ts, long long tr_rs, int step, float sign, int both,
                                  int nblk, const StencilArgs R)
{
    pdl_trigger();
    pdl_wait();
    if ((int)blockIdx.x >= nblk) {   // recording of the input field
        gather_rows(R, blockIdx.x - nblk);
        return;
    }
    const long long sh = blockIdx.y;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= npts * ncorner) return;
    const int j = e / ncorner;
    const long long k = ((long long)sh * npts + j) * ncorner + (e % ncorner);
    const long long p = idx[k];
    const float val = sign * w[k] * traces[sh * tr_ss + (long long)step * tr_ts + j * tr_rs];
    const Pt c = coords(G, p);
    const float sd = damp_at(G, c.x, c.y, c.z);
    const float dd = T.b[p] * val / (1.f + sd);
    for (int f = 0; f < (both ? 2 : 1); f++) {
        atomicAdd(T.d_out + (2 * sh + f) * T.d_out_ss + p, dd);
        atomicAdd(T.u_out + (2 * sh + f) * T.u_out_ss + p, dd);
    }
    if (T.adjoint) {   // the p-field change enters e = E a + S b and f = S a + b
        atomicAdd(T.ef_out + (2 * sh) * T.ef_ss + p, T.E[p] * dd);
        atomicAdd(T.ef_out + (2 * sh + 1) * T.ef_ss + p, T.Sd[p] * dd);
    }
    if (T.img) {
        const float ua = (1.f + sd) * T.h1[(2 * sh) * T.h_ss + p] - (1.f - sd) * T.h0[(2 * sh) * T.h_ss + p];
        atomicAdd(T.img + sh * T.img_ss + p, T.img_scale * ua * dd);
    }
}

// E, S and the tilted axis (ax, ay, az) on the padded layout from the user-layout fields.
__global__ void tti_params_kernel(const GridDev G, const float *eps, const float *delta,
                                  const float *theta, const float *phi, float *E, float *Sd,
                                  float *ax, float *ay, float *az)
{
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < G.Np;
         p += (long long)gridDim.x * blockDim.x) {
        const long long row = p / G.NXp;
        const int x = (int)(p - row * G.NXp);
        if (x >= G.NX) {
            E[p] = Sd[p] = ax[p] = ay[p] = az[p] = 0.f;
            continue;
        }
        const long long u = row * G.NX + x;
        const float th = theta[u], ph = (G.ndim == 3 && phi) ? phi[u] : 0.f;
        E[p] = 1.f + 2.f * eps[u];
        Sd[p] = sqrtf(1.f + 2.f * delta[u]);
        ax[p] = sinf(th) * cosf(ph);
        ay[p] = sinf(th) * sinf(ph);
        az[p] = cosf(th);
    }
}

static unsigned blocks_for(long long n)
{
    const long long g = (n + 255) / 256;
    return (unsigned)(g < 152LL * 32 ? g : 152LL * 32);
}

cudaError_t launch_tti_params(const GridDev &G, const float *eps, const float *delta,
                              const float *theta, const float *phi, float *E, float *Sd,
                              float *ax, float *ay, float *az, cudaStream_t s)
{
    tti_params_kernel<<<blocks_for(G.Np), 256, 0, s>>>(G, eps, delta, theta, phi, E, Sd, ax, ay, az);
    count_launch();
    return cudaGetLastError();
}

// A tiled float map over [w][z][y][x] (rank 4, w_ss floats between w slices, boxes of bw of
// them) or [z][y][x] (rank 3) of a padded field; out-of-range elements read as zero.
static bool tti_map(CUtensorMap *m, const float *base, const GridDev &G, int rank, long long nw, long long w_ss,
                    uint32_t bx, uint32_t by, uint32_t bw = 1)
{
    encode_tiled_fn enc = encoder();
    if (!enc || ((uintptr_t)base & 15) || (w_ss & 3)) return false;
    const cuuint64_t dims[4] = {(cuuint64_t)G.NXp, (cuuint64_t)G.NY, (cuuint64_t)G.NZ, (cuuint64_t)nw};
    const cuuint64_t strides[3] = {(cuuint64_t)G.NXp * 4, (cuuint64_t)G.NXp * G.NY * 4, (cuuint64_t)w_ss * 4};
    const cuuint32_t box[4] = {bx, by, 1, bw};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, (cuuint32_t)rank, (void *)base, dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static int pass2_2d_blocks_per_sm()
{
    static int cached = 0;
    if (!cached) {
        int n = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, tti_pass2_2d_kernel<2, true, false>, 128, 0) != cudaSuccess || n < 1)
            n = 1;
        cached = n;
    }
    return cached;
}

// TX x TY: tile of the marching pass 2; TX x TY1: of pass 1 in 3-D.
template <int TX, int TY, int TY1, bool ADJ>
static cudaError_t tti_passes(const GridDev &G, const TtiArgs &T, cudaStream_t s)
{
    const int ntx = (G.NX + TX - 1) / TX, nty = (G.NY + TY - 1) / TY, nty1 = (G.NY + TY1 - 1) / TY1;
    const long long nv = 2LL * T.nshots;
    const float *xf = ADJ ? T.ef_in : T.u_in;
    const long long xss = ADJ ? T.ef_ss : T.u_in_ss;
    if constexpr (TY == 1) {
        constexpr int ZP1 = 4, ZP2 = 2;
        const long long pairs = G.NXp / 2;
        dim3 grid1((unsigned)((pairs * ((G.NZ + ZP1 - 1) / ZP1) + 127) / 128), T.nshots, 2);
        pdl_launch(tti_pass1_2d_kernel<ZP1>, grid1, 128, 0, s, G, T);
        // Up to two waves the direct pass 2 is the faster one (us a step, direct / marching: 201 x 201
        // 7.7 / 9.6, 401 x 401 8.9 / 11.8, two shots of it 12.3 / 13.5, 801 x 401 12.0 / 13.1; past the
        // line three shots of 401 x 401 and one of 1201 x 401 were equal within 1 %, 16 shots of
        // 1601 x 401 251 / 186).  Both give the same bits.
        const long long blocks = (pairs * ((G.NZ + ZP2 - 1) / ZP2) + 127) / 128;
        if (blocks * T.nshots <= 2LL * device_sm_count() * pass2_2d_blocks_per_sm()) {
            dim3 grid2((unsigned)blocks, T.nshots);
            if (ADJ && T.img) pdl_launch(tti_pass2_2d_kernel<ZP2, true, true>, grid2, 128, 0, s, G, T);
            else pdl_launch(tti_pass2_2d_kernel<ZP2, ADJ, false>, grid2, 128, 0, s, G, T);
            return cudaSuccess;
        }
    }
    // z segments: a march costs its planes and about five more for the z windows' first planes,
    // and a plane time grows with the load (choose_segment): 256^3 takes about 30 (within 2 % of
    // the best of 12 .. 136), one shot of 1601 x 401 6 (17 us a step; with pass 1 marching too
    // 24.5, and 36.7 at the former least of 16).
    const int tz = choose_segment(G.NZ, (double)ntx * nty * T.nshots, (double)device_sm_count() * (TY > 1 ? 4 : 7), 5.0);
    const int nseg = (G.NZ + tz - 1) / tz;
    dim3 grid((unsigned)((long long)ntx * nty * nseg), T.nshots);
    if constexpr (TY > 1) {
        using S1 = Tti1Shape<TX, TY1>;
        const long long ass = T.ay - T.ax;   // a_x, a_y and a_z lie one after the other
        if (T.az - T.ay != ass) return cudaErrorInvalidValue;
        Tti1Maps M1;
        memset(&M1, 0, sizeof M1);
        if (!tti_map(&M1.x, xf, G, 4, nv, xss, S1::WX, S1::WY, 2) ||
            !tti_map(&M1.a, T.ax, G, 4, 3, ass, TX, TY1, 3))
            return cudaErrorInvalidValue;
        cudaFuncSetAttribute(tti_pass1_kernel<TX, TY1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S1::SMEM);
        dim3 grid1((unsigned)((long long)ntx * nty1 * nseg), T.nshots);
        pdl_launch(tti_pass1_kernel<TX, TY1>, grid1, S1::NT, S1::SMEM, s, G, T, tz, ntx, nty1, M1);
    }

    using S2 = Tti2Shape<TX, TY, ADJ>;
    Tti2Maps M;
    memset(&M, 0, sizeof M);
    const long long pss = T.Sd - T.E;   // E, S and dt^2/m lie one after the other
    if (T.b - T.Sd != pss) return cudaErrorInvalidValue;
    bool ok = tti_map(&M.t, T.t, G, 4, nv, T.t_ss, S2::WX, S2::WY, 2) &&
              tti_map(&M.x0, xf, G, 4, nv, xss, S2::WX, S2::WY) &&
              tti_map(&M.ax, T.ax, G, 3, 1, 0, S2::WX, TY) &&
              tti_map(&M.ay, T.ay, G, 3, 1, 0, TX, S2::WY) &&
              tti_map(&M.par, T.E, G, 4, 3, pss, TX, TY, 3) &&
              tti_map(&M.d, T.d_in, G, 4, nv, T.d_in_ss, TX, TY, 2) &&
              tti_map(&M.u, T.u_in, G, 4, nv, T.u_in_ss, TX, TY, S2::NU);
    if (!ok) return cudaErrorInvalidValue;
    auto run = [&](auto kern) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S2::SMEM);
        pdl_launch(kern, grid, S2::NT, S2::SMEM, s, G, T, tz, ntx, nty, M);
    };
    if (ADJ && T.img) run(tti_pass2_kernel<TX, TY, true, true>);
    else run(tti_pass2_kernel<TX, TY, ADJ, false>);
    return cudaSuccess;
}

cudaError_t launch_tti_step(const GridDev &G, const TtiArgs &T, const TtiInject &J, const StencilArgs *rec, cudaStream_t s)
{
    cudaEvent_t ev = prof_begin(PROF_STENCIL, s);
    if (T.img && !T.adjoint) return cudaErrorInvalidValue;   // the imaging condition belongs to the adjoint
    const cudaError_t e = G.ndim == 3 ? (T.adjoint ? tti_passes<32, 8, 16, true>(G, T, s) : tti_passes<32, 8, 16, false>(G, T, s))
                                      : (T.adjoint ? tti_passes<128, 1, 1, true>(G, T, s) : tti_passes<128, 1, 1, false>(G, T, s));
    if (e != cudaSuccess) return e;
    count_launch(2);
    // Recording reads only the step's input, so it shares the injection's launch (a launch of its own,
    // which waited for the step's end, took 2.3 of 13.0 us a step of one shot of 401 x 401).
    const int nblk = (J.npts * J.ncorner + 255) / 256, nrec = rec ? gather_blocks(*rec, 256) : 0;
    if (nblk + nrec > 0) {
        dim3 g2(nblk + nrec, T.nshots);
        pdl_launch(tti_inject_kernel, g2, 256, 0, s, G, T, J.idx, J.w, J.npts, J.ncorner, J.traces, J.tr_ss, J.tr_ts,
                   J.tr_rs, J.step, J.sign, J.both, nblk, rec ? *rec : StencilArgs{});
        count_launch();
    }
    prof_end(PROF_STENCIL, ev, s);
    return cudaGetLastError();
}

}  // namespace wp
