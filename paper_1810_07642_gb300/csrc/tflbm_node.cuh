// Node arithmetic of the fused step in the storage units of
// tflbm_step2.cuh: film pressure, force and collision (Section II of Zitz et
// al., arXiv:1810.07642), written once for X = float2 (two nodes on
// Blackwell's paired FP32 instructions) and X = double (one node).  The
// two- and four-column marches (tflbm_step2.cuh, tflbm_step4.cuh) and the tile
// kernels (tflbm_tile.cuh, tflbm_adjoint_tile.cuh) use it; where a value comes
// from and where a result goes is theirs.
#pragma once
#include "tflbm_step.cuh"

namespace tflbm {

// ---- paired FP32 arithmetic (one instruction for both columns) ------------
__device__ __forceinline__ float2 pk(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 padd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 psub(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float2 pmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

__device__ __forceinline__ float2 pneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 prcp(float2 a) { return make_float2(rcp1(a.x), rcp1(a.y)); }
__device__ __forceinline__ float2 pfdisj(float2 r, int n, int m) { return make_float2(fdisj(r.x, n, m), fdisj(r.y, n, m)); }

// the same names for one FP64 node
__device__ __forceinline__ double padd(double a, double b) { return a + b; }
__device__ __forceinline__ double psub(double a, double b) { return a - b; }
__device__ __forceinline__ double pmul(double a, double b) { return a * b; }
__device__ __forceinline__ double pfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double pneg(double a) { return -a; }
__device__ __forceinline__ double prcp(double a) { return 1.0 / a; }
__device__ __forceinline__ double pfdisj(double r, int n, int m) { return fdisj(r, n, m); }
__device__ __forceinline__ void ptwo_sum(double a, double b, double& s, double& e) { two_sum(a, b, s, e); }

// X: the nodes of one thread; S: their scalar type
template <typename X> struct Lanes;
template <> struct Lanes<float2> {
    using S = float;
    static constexpr int N = 2;
    static __device__ __forceinline__ float2 all(float a) { return make_float2(a, a); }
};
template <> struct Lanes<double> {
    using S = double;
    static constexpr int N = 1;
    static __device__ __forceinline__ double all(double a) { return a; }
};

// Error-free TwoSum on both lanes: a + b = s + e exactly.
__device__ __forceinline__ void ptwo_sum(float2 a, float2 b, float2& s, float2& e)
{
    s = padd(a, b);
    const float2 bb = psub(s, a);
    e = padd(psub(a, psub(s, bb)), psub(b, bb));
}

// ---- pair storage of the moving populations --------------------------------
// V is one aligned pair of stored values; dec gives them as floats in storage
// units (exact), enc rounds two floats to the storage type, dec1 converts one
// stored element.
template <typename SM> struct PairIO;
template <> struct PairIO<float> {
    using V = float2;
    static __device__ __forceinline__ float2 dec(float2 q) { return q; }
    static __device__ __forceinline__ float2 enc(float2 v) { return v; }
    static __device__ __forceinline__ float dec1(float q) { return q; }
};
template <> struct PairIO<double> {
    using V = double;
    static __device__ __forceinline__ double dec(double q) { return q; }
    static __device__ __forceinline__ double enc(double v) { return v; }
    static __device__ __forceinline__ double dec1(double q) { return q; }
};
template <> struct PairIO<__half> {
    using V = __half2;
    static __device__ __forceinline__ float2 dec(__half2 q) { return __half22float2(q); }
    static __device__ __forceinline__ __half2 enc(float2 v) { return __float22half2_rn(v); }
    static __device__ __forceinline__ float dec1(__half q) { return __half2float(q); }
};
template <> struct PairIO<__nv_bfloat16> {
    using V = __nv_bfloat162;
    static __device__ __forceinline__ float2 dec(__nv_bfloat162 q) { return __bfloat1622float2(q); }
    static __device__ __forceinline__ __nv_bfloat162 enc(float2 v) { return __float22bfloat162_rn(v); }
    static __device__ __forceinline__ float dec1(__nv_bfloat16 q) { return __bfloat162float(q); }
};

template <typename V> __device__ __forceinline__ uint32_t bits(V v)
{
    static_assert(sizeof(V) == 4, "16-bit pairs only");
    uint32_t u;
    memcpy(&u, &v, 4);
    return u;
}
template <typename V> __device__ __forceinline__ V from_bits(uint32_t u)
{
    V v;
    memcpy(&v, &u, 4);
    return v;
}
// acc += the two stored values of q, each added to its lane in FP32 by the
// mixed-precision add of sm_100 and later (16-bit operand, FP32 sum, one
// rounding)
template <typename SM> __device__ __forceinline__ void mixed_add(float2& acc, typename PairIO<SM>::V q);
template <> __device__ __forceinline__ void mixed_add<__half>(float2& acc, __half2 q)
{
    unsigned short lo, hi;
    asm("mov.b32 {%0, %1}, %2;" : "=h"(lo), "=h"(hi) : "r"(bits(q)));
    asm("add.rn.f32.f16 %0, %1, %0;" : "+f"(acc.x) : "h"(lo));
    asm("add.rn.f32.f16 %0, %1, %0;" : "+f"(acc.y) : "h"(hi));
}
template <> __device__ __forceinline__ void mixed_add<__nv_bfloat16>(float2& acc, __nv_bfloat162 q)
{
    unsigned short lo, hi;
    asm("mov.b32 {%0, %1}, %2;" : "=h"(lo), "=h"(hi) : "r"(bits(q)));
    asm("add.rn.f32.bf16 %0, %1, %0;" : "+f"(acc.x) : "h"(lo));
    asm("add.rn.f32.bf16 %0, %1, %0;" : "+f"(acc.y) : "h"(hi));
}

// A 3 x 3 stencil window: for each of the rows n (+y), c, s (-y) the values
// at the thread's own columns and the ones to the left and right of them.
template <typename X>
struct Win {
    X n0, nL, nR, c0, cL, cR, s0, sL, sR;
};

// ---------------------------------------------------------------------------
// Node arithmetic.

// Film pressure (Eq. pfilm with Eq. disjoiningP) from the h window; writes 1/h
// to ih.
template <typename X>
__device__ __forceinline__ X node_pressure(const Win<X>& H, X kap, bool disj, const Consts<typename Lanes<X>::S>& C,
                                           X& ih)
{
    using S = typename Lanes<X>::S;
    auto pk = [](S a) { return Lanes<X>::all(a); };
    // Eq. (n_laplace): axis neighbours left + right + up + down, diagonal the four corners
    const X axis = padd(padd(H.cL, H.cR), padd(H.n0, H.s0));
    const X diag = padd(padd(H.nL, H.nR), padd(H.sL, H.sR));
    // the large terms cancel in the last fma, exactly but for the rounding of
    // 4 axis + diag; with -20 c0 + diag rounded first, heights after 60 steps of a
    // 700^2 drop were 1.15 times as far from FP64 (1.48e-7 against 1.29e-7)
    X lap = pmul(pfma(pk(-S(20.0)), H.c0, pfma(pk(S(4.0)), axis, diag)), pk(S(1.0 / 6.0)));
    const X h = padd(H.c0, pk(C.href));
    ih = prcp(h);
    if (disj) {
        const X r = pmul(pk(C.hstar), ih);
        X fd;
        if (C.n_exp == 3 && C.m_exp == 2) fd = pmul(pmul(r, r), psub(r, pk(S(1.0))));
        else fd = pfdisj(r, C.n_exp, C.m_exp);
        lap = pfma(pmul(pk(C.pi_sgn), kap), fd, lap);
    }
    return pmul(pk(-C.gamma), lap);
}

// The total force at a node, the velocity u and the momentum e of the
// equilibria (Eqs. force, forcefric, alphafric).  P: the p window (n = row o+1,
// s = row o-1).
template <typename X>
__device__ __forceinline__ void node_force(const Win<X>& P, X h, X ih, X jx, X jy, const Consts<typename Lanes<X>::S>& C,
                                           X& ux, X& uy, X& ex, X& ey, X& Fx, X& Fy)
{
    using S = typename Lanes<X>::S;
    auto pk = [](S a) { return Lanes<X>::all(a); };
    // Eq. (derivative): grad p = 3 sum_l w_l c_l p(x + c_l)
    const X gpx = pfma(psub(P.cR, P.cL), pk(S(1.0 / 3.0)),
                       pmul(padd(psub(P.nR, P.nL), psub(P.sR, P.sL)), pk(S(1.0 / 12.0))));
    const X gpy = pfma(psub(P.n0, P.s0), pk(S(1.0 / 3.0)),
                       pmul(padd(psub(P.nR, P.sR), psub(P.nL, P.sL)), pk(S(1.0 / 12.0))));
    // nu alpha u = 6 nu j / (2h^2 + 6 delta h + 3 delta^2)
    const X den = pfma(h, pfma(pk(S(2.0)), h, pk(S(6.0) * C.delta)), pk(S(3.0) * C.delta * C.delta));
    const X fr = pmul(pk(C.nu6), prcp(den));
    // Eq. (LBE) as printed: u = j/h.  Second-order forcing (C.forcing):
    // u (h + nu alpha/2) = j + F'/2 and the equilibria use h u for j (see
    // collide_store)
    if (C.forcing) {
        const X fpx = pmul(h, psub(pk(C.gx), gpx)), fpy = pmul(h, psub(pk(C.gy), gpy));
        const X d = pfma(pk(S(0.5)), fr, pk(S(1.0)));
        const X q = pmul(ih, prcp(d));
        ux = pmul(pfma(pk(S(0.5)), fpx, jx), q);
        uy = pmul(pfma(pk(S(0.5)), fpy, jy), q);
        ex = pmul(h, ux);
        ey = pmul(h, uy);
        Fx = psub(fpx, pmul(fr, ex));
        Fy = psub(fpy, pmul(fr, ey));
    } else {
        Fx = psub(pmul(h, psub(pk(C.gx), gpx)), pmul(fr, jx));
        Fy = psub(pmul(h, psub(pk(C.gy), gpy)), pmul(fr, jy));
        ux = pmul(jx, ih);
        uy = pmul(jy, ih);
        ex = jx;
        ey = jy;
    }
}

// Eq. (equilibria) with e^2 = 1 as S +- D per opposite pair; the even parts S in
// storage units, (S - R_l) ms.
template <typename SM, typename X>
__device__ __forceinline__ void node_even(X h, X ux, X uy, X ex, X ey, const Consts<typename Lanes<X>::S>& C, X& Sx,
                                          X& Sy, X& Sa, X& Sb)
{
    using S = typename Lanes<X>::S;
    auto pk = [](S a) { return Lanes<X>::all(a); };
    constexpr bool NARROW = sizeof(SM) == 2;
    // storage scale (1 for full-width storage, a compile-time constant there)
    const S ms = NARROW ? C.mscale : S(1);
    // A6 = 6 A = h (g h - u^2)
    const X A6 = pmul(h, psub(pmul(pk(C.g), h), pfma(ux, ux, pmul(uy, uy))));
    const X Aa = NARROW ? pfma(A6, pk(ms * S(1.0 / 6.0)), pk(C.nr_axis)) : pmul(A6, pk(S(1.0 / 6.0)));
    const X Ad = NARROW ? pfma(A6, pk(ms * S(1.0 / 24.0)), pk(C.nr_diag)) : pmul(A6, pk(S(1.0 / 24.0)));
    Sx = pfma(pmul(ex, pk(S(0.5) * ms)), ux, Aa);
    Sy = pfma(pmul(ey, pk(S(0.5) * ms)), uy, Aa);
    const X a = padd(ux, uy), b = psub(uy, ux);
    const X h8 = pmul(h, pk(S(0.125) * ms));
    Sa = pfma(pmul(h8, a), a, Ad);
    Sb = pfma(pmul(h8, b), b, Ad);
}

// Post-collision moving populations at omega = 1: the even parts and the odd
// parts of G = e + F (source 3 w_l c_l . F), in storage units; o[l - 1].
template <typename SM, typename X>
__device__ __forceinline__ void node_odd(X Sx, X Sy, X Sa, X Sb, X Gx, X Gy, const Consts<typename Lanes<X>::S>& C,
                                         X (&o)[8])
{
    using S = typename Lanes<X>::S;
    const S ms = sizeof(SM) == 2 ? C.mscale : S(1);
    const X m3 = Lanes<X>::all(ms * S(1.0 / 3.0)), m12 = Lanes<X>::all(ms * S(1.0 / 12.0));
    const X Dx = pmul(Gx, m3), Dy = pmul(Gy, m3);
    const X Da = pmul(padd(Gx, Gy), m12), Db = pmul(psub(Gy, Gx), m12);
    o[0] = padd(Sx, Dx); o[4] = psub(Sx, Dx);
    o[2] = padd(Sy, Dy); o[6] = psub(Sy, Dy);
    o[1] = padd(Sa, Da); o[5] = psub(Sa, Da);
    o[3] = padd(Sb, Db); o[7] = psub(Sb, Db);
}

// Stored rest population f*_0 - href = (h - href) - sum_{l>0} f*_l, with the
// exact residuals (er: of the pull sum) folded back into f_1 and f_5 as in
// collide_store; full-width storage.
template <typename X>
__device__ __forceinline__ X node_fold(X dh, X er, X (&o)[8])
{
    const X osum = padd(padd(padd(o[0], o[4]), padd(o[2], o[6])), padd(padd(o[1], o[5]), padd(o[3], o[7])));
    X o0, e2;
    ptwo_sum(dh, pneg(osum), o0, e2);
    const X half_r = pmul(padd(er, e2), Lanes<X>::all(typename Lanes<X>::S(0.5)));
    o[0] = padd(o[0], half_r);
    o[4] = padd(o[4], half_r);
    return o0;
}

// The same for 16-bit storage: q receives the stored values.
template <typename SM>
__device__ __forceinline__ float2 node_fold_narrow(float2 dh, float2 er, const float2 (&o)[8], const Consts<float>& C,
                                                   typename PairIO<SM>::V (&q)[8])
{
    using IO = PairIO<SM>;
    using V = typename IO::V;
    const V q1r = IO::enc(o[0]);
#pragma unroll
    for (int l = 1; l < 8; ++l) q[l] = IO::enc(o[l]);
    // what the readers reconstruct of l = 2..8 (storage units; each stored
    // value enters the FP32 sum by a mixed-precision add, which takes the
    // 16-bit operand as it is), summed so that exchanging +y and -y (a march
    // the other way) gives the same bits
    float2 r28 = IO::dec(q[1]), r37 = IO::dec(q[2]), r46 = IO::dec(q[3]);
    mixed_add<SM>(r28, q[7]);
    mixed_add<SM>(r37, q[6]);
    mixed_add<SM>(r46, q[5]);
    float2 rest = padd(padd(r28, r46), r37);
    mixed_add<SM>(rest, q[4]);
    float2 rest1 = rest;
    mixed_add<SM>(rest1, q1r);
    // the moving populations' total with f_1 unrounded and rounded
    const float2 osum = pfma(padd(rest, o[0]), pk(C.minv), pk(C.r_sum));
    const float2 osr = pfma(rest1, pk(C.minv), pk(C.r_sum));
    // the last residual goes to the finer of the two roundings: the 16-bit
    // one of f_1 - R or the FP32 one of f_0 - href (see collide_store)
    constexpr float kRatio = std::is_same<SM, __half>::value ? 8192.0f : 65536.0f;
    const float kr = kRatio * C.minv;  // |f_1 - R| = |o1| / ms
    const bool lx = fabsf(o[0].x) * kr < fabsf(dh.x - osum.x);
    const bool ly = fabsf(o[0].y) * kr < fabsf(dh.y - osum.y);
    const float2 os = make_float2(lx ? osum.x : osr.x, ly ? osum.y : osr.y);
    float2 o0v, e2, o0n, e3;
    ptwo_sum(dh, pneg(os), o0v, e2);
    ptwo_sum(o0v, padd(er, e2), o0n, e3);
    const V q1l = IO::enc(pfma(e3, pk(C.mscale), o[0]));
    const uint32_t mask = (lx ? 0x0000ffffu : 0u) | (ly ? 0xffff0000u : 0u);
    q[0] = from_bits<V>((bits(q1l) & mask) | (bits(q1r) & ~mask));
    return o0n;
}

// Force and collision (the arithmetic of collide_store on every lane, in
// storage units).  f: the pulled moving populations in storage units, fstride
// apart (omega != 1 only).  The post-collision populations go to
// store(f_0 - href, q[8]), q as stored.
template <typename SM, bool OMEGA1, typename X, typename Store>
__device__ __forceinline__ void node_collide(const Win<X>& P, X dh, X ih, X jx, X jy, X er, const X* f, int fstride,
                                             const Consts<typename Lanes<X>::S>& C, Store store)
{
    using S = typename Lanes<X>::S;
    auto pk = [](S a) { return Lanes<X>::all(a); };
    constexpr bool NARROW = sizeof(SM) == 2;
    const S ms = NARROW ? C.mscale : S(1);
    const X h = padd(dh, pk(C.href));
    X ux, uy, ex, ey, Fx, Fy, Sx, Sy, Sa, Sb;
    node_force(P, h, ih, jx, jy, C, ux, uy, ex, ey, Fx, Fy);
    node_even<SM>(h, ux, uy, ex, ey, C, Sx, Sy, Sa, Sb);
    // second-order source: odd part scaled by (1 - omega/2), even part T
    X Tx = pk(S(0.0)), Ty = pk(S(0.0)), Ta = pk(S(0.0)), Tb = pk(S(0.0));
    if (C.forcing) {
        const X ks = pk(S(1.0) - S(0.5) * C.omega), a = padd(ux, uy), b = psub(uy, ux);
        Fx = pmul(Fx, ks);
        Fy = pmul(Fy, ks);
        const X uF3 = pmul(pfma(ux, Fx, pmul(uy, Fy)), pk(ms * S(1.0 / 3.0)));
        Tx = pfma(pmul(ux, Fx), pk(ms), pneg(uF3));
        Ty = pfma(pmul(uy, Fy), pk(ms), pneg(uF3));
        Ta = pmul(pfma(pmul(a, padd(Fx, Fy)), pk(ms), pneg(uF3)), pk(S(0.25)));
        Tb = pmul(pfma(pmul(b, psub(Fy, Fx)), pk(ms), pneg(uF3)), pk(S(0.25)));
        if constexpr (OMEGA1) {
            Sx = padd(Sx, Tx);
            Sy = padd(Sy, Ty);
            Sa = padd(Sa, Ta);
            Sb = padd(Sb, Tb);
        }
    }
    X o[8];
    if constexpr (OMEGA1) {
        node_odd<SM>(Sx, Sy, Sa, Sb, padd(ex, Fx), padd(ey, Fy), C, o);
    } else {
        // (1 - omega)(f_l - R_l) + omega (f_eq_l - R_l) + source, in storage
        // units: (1 - omega) f_l + V +- E per opposite pair, V = omega S + T, E
        // the odd parts of omega e + F
        const X w = pk(C.omega), m = pk(S(1.0) - C.omega);
        const X m3 = pk(ms * S(1.0 / 3.0)), m12 = pk(ms * S(1.0 / 12.0));
        const X Gx = pfma(w, ex, Fx), Gy = pfma(w, ey, Fy);
        auto opposite = [&](X s, X t, X e, int l) {  // populations l + 1 and l + 5
            const X v = pfma(w, s, t);
            o[l] = pfma(m, f[l * fstride], padd(v, e));
            o[l + 4] = pfma(m, f[(l + 4) * fstride], psub(v, e));
        };
        opposite(Sx, Tx, pmul(Gx, m3), 0);
        opposite(Sa, Ta, pmul(padd(Gx, Gy), m12), 1);
        opposite(Sy, Ty, pmul(Gy, m3), 2);
        opposite(Sb, Tb, pmul(psub(Gy, Gx), m12), 3);
    }
    if constexpr (!NARROW) {
        const X o0 = node_fold(dh, er, o);
        store(o0, o);
    } else {
        typename PairIO<SM>::V q[8];
        const X o0 = node_fold_narrow<SM>(dh, er, o, C, q);
        store(o0, q);
    }
}

// Moments from the sums of pulled populations in storage units: f0 - href;
// Rs, Ls the populations arriving from the left (l = 1, 2, 8) and the right (l
// = 5, 4, 6), s26 those along y (l = 3, 7), jyr their y momentum.  dh = h -
// href: the moving total is small, the last addition is error-free (see sum9).
template <typename SM, typename X>
__device__ __forceinline__ void node_moments(X f0, X Rs, X Ls, X s26, X jyr, const Consts<typename Lanes<X>::S>& C,
                                             X& dh, X& er, X& jx, X& jy)
{
    const X tot = padd(s26, padd(Rs, Ls));
    if constexpr (sizeof(SM) == 2) {
        const X minv = Lanes<X>::all(C.minv);
        ptwo_sum(f0, pfma(tot, minv, Lanes<X>::all(C.r_sum)), dh, er);
        jx = pmul(psub(Rs, Ls), minv);
        jy = pmul(jyr, minv);
    } else {
        ptwo_sum(f0, tot, dh, er);
        jx = psub(Rs, Ls);
        jy = jyr;
    }
}

}  // namespace tflbm
