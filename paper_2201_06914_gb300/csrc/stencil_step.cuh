// One time step of the isotropic scheme at four adjacent columns, shared by the
// single-step (stencil.cu) and two-step (stencil2.cu) kernels so that both perform the
// same operations in the same order and give the same bits.
//
// The arithmetic runs on pairs of columns with the packed FP32 instructions of sm_100+
// (add/sub/mul/fma .rn.f32x2: each lane is the IEEE single-precision operation with
// round-to-nearest), which halves the instruction count of the Laplacian.
//
// Laplacian in pairwise form with the axes merged (Sec. 2.1, space order 8):
//   L u = (1/hx^2) sum_k c_k ( (u[x+k] + u[x-k]) + rz (u[z+k] + u[z-k]) + ry (u[y+k] + u[y-k])
//                              - 2 (1 + rz + ry) u )
// with rz = hx^2/hz^2, ry = hx^2/hy^2.  Neighbour pairs are summed first and the centre is
// removed per offset, which keeps the FP32 rounding of L u at the level of the fully
// differenced form (the plain sum c_0 u + sum c_k (u[+k] + u[-k]) loses about a digit on
// smooth fields).  Then, with s = sigma dt / 2 and b = dt^2 / m, the (u, d) form (adjoint)
//   d^{n+1} = d^n + b (L u + q)                               (s = 0)
//   d^{n+1} = ((1 - s) d^n + b (L u + q)) * rcp(1 + s)        (absorbing layer)
//   u^{n+1} = u^n + d^{n+1}
// or the (w, d) form (forward), whose state is w^{n-1} = L u^{n-1} and d^n = u^n - u^{n-1}
// and which never forms u:
//   w^n     = w^{n-1} + L d^n
//   d^{n+1} = d^n + b (w^n + q)                               (s = 0)
//   d^{n+1} = ((1 - s) d^n + b (w^n + q)) * rcp(1 + s)        (absorbing layer)
// Both are the same recurrence in exact arithmetic (L is linear).  In FP32 the (w, d) form
// never rounds u itself: the (u, d) form adds d to a much larger u every step, and L
// amplifies that rounding noise (white in space) far more than it amplifies the wave, so
// u_tt = b (w + q) / dt^2, which the forward's probe projections are built from, is
// several times more accurate in the (w, d) form (2.9e-6 instead of 1.5e-5 relative L2
// for P_u after 1000 steps of the two-layer 201 x 201 workload, FP32 emulation on the
// CPU).  The adjoint keeps the (u, d) form: its projections use v itself, not a second
// derivative.
//
// In both forms the field that the stencil reads with halos ("X": u, or d) and the field
// read only at the own point ("Y": d, or w) enter and leave through the same arguments:
// cc/wz = X^n, din = Y^n, un = X^{n+1}, dn = Y^{n+1}.
#pragma once

#include "wp_internal.cuh"

namespace wp {
namespace step {

typedef unsigned long long f2;   // two floats in one 64-bit register (low word first)

struct __align__(16) P4 {        // four adjacent columns as two pairs
    f2 a, b;                     // columns (0, 1) and (2, 3)
};

__device__ __forceinline__ f2 pk(float lo, float hi)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void upk(f2 v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f2 add2(f2 a, f2 b)
{
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b)
{
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b)
{
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c)
{
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f2 dup(float v) { return pk(v, v); }

__device__ __forceinline__ P4 lds(uint32_t addr)
{
    P4 v;
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(v.a), "=l"(v.b) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts(uint32_t addr, const P4 &v)
{
    asm volatile("st.shared.v2.b64 [%0], {%1, %2};" ::"r"(addr), "l"(v.a), "l"(v.b) : "memory");
}
__device__ __forceinline__ P4 zero() { return P4{0ull, 0ull}; }

__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ const f2 &half(const P4 &v, int p) { return p == 0 ? v.a : v.b; }

// Sums of the x neighbours +k and -k of the thread's four columns, pair by pair, from the 12
// values wl | centre | wr.  Even offsets are aligned pairs (one packed add); odd offsets would
// need both operands re-paired with register moves first, so they are two scalar adds instead:
// the same IEEE additions.
__device__ __forceinline__ f2 xsum(const P4 &wl, const P4 &cc, const P4 &wr, int p, int k)
{
    const int ip = 4 + 2 * p + k, im = 4 + 2 * p - k;   // first column of either operand
    auto quad = [&](int i) -> const P4 & { return i < 4 ? wl : i < 8 ? cc : wr; };
    if ((k & 1) == 0) return add2(half(quad(ip), (ip & 3) >> 1), half(quad(im), (im & 3) >> 1));
    auto col = [&](int i) {
        float lo, hi;
        upk(half(quad(i), (i & 3) >> 1), lo, hi);
        return (i & 1) ? hi : lo;
    };
    return pk(__fadd_rn(col(ip), col(im)), __fadd_rn(col(ip + 1), col(im + 1)));
}

// The step's constants as packed pairs (both halves equal): hx^2/hz^2, hx^2/hy^2, -2 (1 + rz +
// ry), 1/hx^2 and the weights of offsets 1..4.  A packed instruction takes a constant only from
// a register pair; built from immediates or kernel parameters the compiler re-creates the pair
// with two moves at every use, so a kernel reads them once from shared memory (values the
// compiler cannot re-create) and they stay in registers.
struct Coef {
    f2 rz, ry, nk, ih, c[4];
};
__device__ __forceinline__ void coef_store(f2 (*sm)[8], const GridDev &G)   // one thread, before a barrier
{
    const float v[8] = {G.lrz, G.lry, -G.lapK, G.ihx2, WP_C1, WP_C2, WP_C3, WP_C4};
#pragma unroll
    for (int i = 0; i < 8; i++) (*sm)[i] = dup(v[i]);
}
__device__ __forceinline__ Coef coef_load(f2 (*sm)[8])
{
    f2 v[8];
#pragma unroll
    for (int i = 0; i < 8; i++)
        asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v[i]) : "r"((uint32_t)__cvta_generic_to_shared(&(*sm)[i])));
    return Coef{v[0], v[1], v[2], v[3], {v[4], v[5], v[6], v[7]}};
}

// hx^2 times the Laplacian of one pair of columns: zs[k - 1], ys[k - 1] are the sums of the z and y neighbours
// +k and -k (ys only if Y).
template <bool Y>
__device__ __forceinline__ f2 lap_pair(const P4 &wl, const P4 &cc, const P4 &wr, int p, const f2 zs[RAD],
                                       const f2 ys[RAD], const Coef &K)
{
    const f2 c = half(cc, p);
    f2 acc = 0ull;
#pragma unroll
    for (int k = 1; k <= RAD; k++) {
        f2 sp = fma2(K.rz, zs[k - 1], xsum(wl, cc, wr, p, k));
        if (Y) sp = fma2(K.ry, ys[k - 1], sp);
        // centre removed with one rounding: sp - 2 (1 + rz + ry) u (the neighbour sum and
        // the centre term nearly cancel on smooth fields)
        const f2 t = fma2(K.nk, c, sp);
        acc = k == 1 ? mul2(K.c[k - 1], t) : fma2(K.c[k - 1], t, acc);
    }
    return acc;
}

// Update of the four columns from acc = hx^2 L u.  cc: own columns of X; din: of Y; sqv:
// injected terms (read if inj); sdx: absorbing-layer term of the columns along x (and y); z:
// plane index.  `interior` may be false where the absorbing term is zero: the layer's form then
// multiplies by 1 - 0 and by rcp(1) = 1 and gives the same bits.  Returns the new increment and
// field; sdv receives the absorbing term of each column (0 inside).
//
// The assembler may contract a packed multiply that feeds a packed add into one fma (also with
// .rn), differently in each kernel.  Wherever a product meets a sum, this routine therefore
// either asks for the fma or multiplies the halves with scalar .rn instructions, which are
// never contracted, so that every kernel gives the same bits.
template <bool WD>
__device__ __forceinline__ void update4(const P4 &cc, const f2 acc[2], const P4 &din, const P4 &bb, const float *sqv,
                                        bool inj, bool interior, const float sdx[4], int z, const GridDev &G,
                                        const Coef &K, P4 &dn, P4 &un, float sdv[4])
{
    f2 wn[2], lap[2];
#pragma unroll
    for (int p = 0; p < 2; p++) {
        if (WD) {
            // w^n = w^{n-1} + L d^n; the source enters b (w^n + q) below
            lap[p] = wn[p] = fma2(K.ih, acc[p], half(din, p));
            if (inj) lap[p] = add2(lap[p], pk(sqv[2 * p], sqv[2 * p + 1]));
        } else {
            lap[p] = mul2(K.ih, acc[p]);
            if (inj) {
                float a0, a1, k0, k1;
                upk(acc[p], a0, a1);
                upk(K.ih, k0, k1);
                lap[p] = add2(pk(__fmul_rn(k0, a0), __fmul_rn(k1, a1)), pk(sqv[2 * p], sqv[2 * p + 1]));
            }
        }
    }
    // the increment the update starts from: d^n (the own column of X in the (w, d) form)
    const P4 &dprev = WD ? cc : din;
    f2 d[2];
    if (interior) {
        d[0] = fma2(bb.a, lap[0], dprev.a);
        d[1] = fma2(bb.b, lap[1], dprev.b);
#pragma unroll
        for (int j = 0; j < 4; j++) sdv[j] = 0.f;
    } else {
        const float sdz = damp_term(z, G.nz, G.nbl, G.hs0z, G.inv_nbl);
        const f2 one = dup(1.f);
#pragma unroll
        for (int p = 0; p < 2; p++) {
            const f2 sd = add2(pk(sdx[2 * p], sdx[2 * p + 1]), dup(sdz));
            const f2 t = fma2(half(bb, p), lap[p], mul2(sub2(one, sd), half(dprev, p)));
            float o0, o1;
            upk(add2(one, sd), o0, o1);
            float t0, t1;
            upk(t, t0, t1);
            d[p] = pk(__fmul_rn(t0, rcp_approx(o0)), __fmul_rn(t1, rcp_approx(o1)));
            upk(sd, sdv[2 * p], sdv[2 * p + 1]);
        }
    }
    if (WD) {
        un.a = d[0];   // X^{n+1} = d^{n+1}
        un.b = d[1];
        dn.a = wn[0];  // Y^{n+1} = w^n
        dn.b = wn[1];
    } else {
        dn.a = d[0];
        dn.b = d[1];
        un.a = add2(cc.a, d[0]);
        un.b = add2(cc.b, d[1]);
    }
}

// One step at the four columns of the thread.  wz: own column z window with the centre at
// wz[RAD]; wy_p / wy_m: y neighbours +k / -k (3-D only, Y = true); wl / wr: x neighbours
// (columns -4..-1 and +4..+7).
template <bool Y, bool WD = false>
__device__ __forceinline__ void step4(const P4 *wz, const P4 *wy_p, const P4 *wy_m, const P4 &wl,
                                      const P4 &wr, const P4 &din, const P4 &bb, const float *sqv,
                                      bool inj, bool interior, const float sdx[4], int z,
                                      const GridDev &G, const Coef &K, P4 &dn, P4 &un, float sdv[4])
{
    f2 acc[2];
#pragma unroll
    for (int p = 0; p < 2; p++) {
        f2 zs[RAD], ys[RAD];
#pragma unroll
        for (int k = 1; k <= RAD; k++) {
            zs[k - 1] = add2(half(wz[RAD + k], p), half(wz[RAD - k], p));
            ys[k - 1] = Y ? add2(half(wy_p[k - 1], p), half(wy_m[k - 1], p)) : 0ull;
        }
        acc[p] = lap_pair<Y>(wl, wz[RAD], wr, p, zs, ys, K);
    }
    update4<WD>(wz[RAD], acc, din, bb, sqv, inj, interior, sdx, z, G, K, dn, un, sdv);
}

}  // namespace step
}  // namespace wp
