// Fused adjoint of one thin-film step in tiles (the transpose of the phases
// listed in tflbm_adjoint.cu, evaluated in one pass over the lattice).
//
// What it reads.  The step depends on its state f(t) beyond the linear factor
// (1 - omega) only through h and j, so the tape keeps those three fields a step
// (12 B a node in FP32, not 36) and the adjoint never pulls populations.  At
// omega = 1 the adjoint state has three fields as well: a_l(t) = aH + c_l . aJ,
// stored as (aH, aJ_x, aJ_y); otherwise a_l(t) = aH + c_l . aJ + (1 - omega) mu_l
// keeps nine.  Per node and step in FP32 at omega = 1: 12 B of moments, 12 B in
// and 12 B out of adjoint state, kappa and the read-modify-write of dL/dkappa,
// 48 B in place of the 120 B of populations and nine-plane adjoints.
//
// What bounds it.  On lattices that L2 holds (the usual case for a gradient:
// 512^2) the round trips: the four nested radius-1 stencils (h -> p -> grad p
// and -h aF -> transposed gradient -> Laplacian) were a march of 15 rows for
// bands of 4; a tile has three barriers a step (one more than the forward
// tile, for the a(t+1) neighbourhood in shared memory):
//   1  a(t+1) of the tile and a halo of 3 (omega = 1), h of the halo of 2
//   2  with mu_l = a_l(x + c_l, t+1): ag = -h aF on the halo of 2; on the tile
//      the equilibrium and source adjoints
//   3  p and -gamma ap (transposed gradient of ag) on the halo of 1; on the
//      tile the disjoining-pressure adjoint and dL/dkappa
//   4  on the tile grad p, the force adjoint, the Laplacian of -gamma ap, a(t)
// 512^2 FP32, a gradient of 400 steps: 23.8 ms as marches of populations, 6.1 now,
// of which an adjoint step took 27 us, 9 now (820 instructions a warp,
// half of the issue slots; 512 tiles on 152 SMs); threads, lanes, tiles and the
// treatment of the edges are those of tflbm_tile.cuh.
#pragma once
#include "tflbm_tile.cuh"

namespace tflbm {

__device__ __forceinline__ float2 operator+(float2 a, float2 b) { return padd(a, b); }
__device__ __forceinline__ float2 operator-(float2 a, float2 b) { return psub(a, b); }
__device__ __forceinline__ float2 operator*(float2 a, float2 b) { return pmul(a, b); }
__device__ __forceinline__ float2 pipow(float2 r, int n) { return make_float2(ipow(r.x, n), ipow(r.y, n)); }
__device__ __forceinline__ double pipow(double r, int n) { return ipow(r, n); }

// mom: (h - href, j_x, j_y) of the state f(t), [3][ny][nx], and whether the
// launch before this one may still be writing it (fresh); early: let the next
// step's CTAs in a phase earlier; an, a: a(t+1) and
// a(t), [3][ny][nx] at omega = 1, else [9][ny][nx]; gk += dL/dkappa.
template <typename S, int TX, int TY, bool OMEGA1, int RESIDENT>
__global__ void __launch_bounds__(TX* TY / Lanes<typename TileX<S>::X>::N, RESIDENT / (TX * TY / Lanes<typename TileX<S>::X>::N))
k_adjoint_tile(const S* __restrict__ mom, bool fresh, bool early, const S* __restrict__ an, S* __restrict__ a,
               S* __restrict__ gk, const S* __restrict__ kappa, const Geom G, const Consts<S> C)
{
    using X = typename TileX<S>::X;
    constexpr int N = Lanes<X>::N, NT = TX * TY / N, HALF = TY / N;
    constexpr int HW = TX + 4, PW = TX + 2, AW = TX + 6;
    constexpr int HN = HW * (TY + 4) - TX * TY, PN = PW * (TY + 2) - TX * TY;
    constexpr int HP = HN / N, PP = PN / N;
    static_assert(HN % N == 0 && PN % N == 0 && TY % N == 0, "halo nodes come in whole groups");
    static_assert(HP <= NT && PP <= NT, "one group of halo nodes a thread");
    __shared__ S hs[TY + 4][HW];                    // h - href; tile node (c, r) at [r + 2][c + 2]
    __shared__ S gxs[TY + 4][HW], gys[TY + 4][HW];  // ag, same places
    __shared__ S ps[TY + 2][PW], ls[TY + 2][PW];    // p and -gamma ap; tile node at [r + 1][c + 1]
    __shared__ S as[OMEGA1 ? 3 : 1][OMEGA1 ? TY + 6 : 1][OMEGA1 ? AW : 1];  // a(t+1); tile node at [r + 3][c + 3]

    const int t = threadIdx.x, nx = G.nx, ny = G.ny;
    const long long n = (long long)nx * ny;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int c = t % TX, r = t / TX;  // own nodes: (c, r + k HALF)
    const bool disj = kappa != nullptr || C.kappa_u != S(0);
    auto pk = [](S v) { return Lanes<X>::all(v); };
    auto node = [&](int cc, int rr) {
        return TFLBM_IDX(ring_index(y0 + rr, ny) * nx + ring_index(x0 + cc, nx), n, C.status);
    };
    // offset k within a plane of an or a
    auto in_plane = [&](uint32_t k) { return TFLBM_IDX(k, n, C.status); };
    auto lanes = [&](auto fn) {
        fn(std::integral_constant<int, 0>{});
        if constexpr (N == 2) fn(std::integral_constant<int, 1>{});
    };

    // ---- 1: every load of the step is requested before any is waited for; the
    // record and kappa, which no adjoint step writes, before the step at t + 1 ends
    if (fresh) dependent_launch_wait();
    X dh, jx, jy, kap, gold, kh;
    lanes([&](auto k_c) {
        constexpr int K = decltype(k_c)::value;
        const int i = node(c, r + K * HALF);
        lane_of<K>(dh) = ldro(mom + i);
        lane_of<K>(jx) = ldro(mom + n + i);
        lane_of<K>(jy) = ldro(mom + 2 * n + i);
        lane_of<K>(kap) = kappa ? ldro(kappa + i) : C.kappa_u;
    });
    X hh;  // halo nodes of h: h - href, then h
    int hc[N], hr[N], pc[N], pr[N];
    if (t < HP) {
        lanes([&](auto k_c) {
            constexpr int K = decltype(k_c)::value;
            tile_halo<TX, TY, 2>(t + K * HP, hc[K], hr[K]);
            lane_of<K>(hh) = ldro(mom + node(hc[K], hr[K]));
        });
    }
    if (t < PP) {
        lanes([&](auto k_c) {
            constexpr int K = decltype(k_c)::value;
            tile_halo<TX, TY, 1>(t + K * PP, pc[K], pr[K]);
            lane_of<K>(kh) = kappa ? ldro(kappa + node(pc[K], pr[K])) : C.kappa_u;
        });
    }
    dependent_launch_wait();
    lanes([&](auto k_c) {
        constexpr int K = decltype(k_c)::value;
        lane_of<K>(gold) = gk[node(c, r + K * HALF)];
    });
    if constexpr (OMEGA1) {
        // the tile's columns, NT / TX rows a pass, then the three on either side
        constexpr int RP = NT / TX, PASSES = (TY + 6 + RP - 1) / RP, SIDES = (6 * (TY + 6) + NT - 1) / NT;
        S v[PASSES + SIDES][3];
        const uint32_t xc = ring_index(x0 + c, nx);
#pragma unroll
        for (int p = 0; p < PASSES; ++p) {
            const int rr = r + p * RP;
            const uint32_t k = in_plane(ring_index(y0 + rr - 3, ny) * nx + xc);
#pragma unroll
            for (int f = 0; f < 3; ++f) v[p][f] = rr < TY + 6 ? ldro(an + f * n + k) : S(0);
        }
#pragma unroll
        for (int p = 0; p < SIDES; ++p) {
            const int i = t + p * NT, rr = i / 6, cc = i % 6 < 3 ? i % 6 - 3 : TX + i % 6 - 3;
            const uint32_t k = node(cc, rr - 3);
#pragma unroll
            for (int f = 0; f < 3; ++f) v[PASSES + p][f] = rr < TY + 6 ? ldro(an + f * n + k) : S(0);
        }
#pragma unroll
        for (int p = 0; p < PASSES + SIDES; ++p) {
            const int i = t + (p - PASSES) * NT;
            const int rr = p < PASSES ? r + p * RP : i / 6;
            const int cc = p < PASSES ? c : (i % 6 < 3 ? i % 6 - 3 : TX + i % 6 - 3);
            if (rr < TY + 6) {
#pragma unroll
                for (int f = 0; f < 3; ++f) as[f][rr][cc + 3] = v[p][f];
            }
        }
    }
    lanes([&](auto k_c) {
        constexpr int K = decltype(k_c)::value;
        hs[r + K * HALF + 2][c + 2] = lane_of<K>(dh);
        if (t < HP) hs[hr[K] + 2][hc[K] + 2] = lane_of<K>(hh);
    });
    __syncthreads();

    // ---- 2: mu_l of the node at tile position (cc, rr), into lane K
    auto gather = [&](auto k_c, int cc, int rr, X (&mu)[9]) {
        constexpr int K = decltype(k_c)::value;
        if constexpr (OMEGA1) {
            auto at = [&](int f, int dx, int dy) { return as[f][rr + 3 + dy][cc + 3 + dx]; };
            lane_of<K>(mu[0]) = at(0, 0, 0);
            lane_of<K>(mu[1]) = at(0, 1, 0) + at(1, 1, 0);
            lane_of<K>(mu[2]) = at(0, 1, 1) + (at(1, 1, 1) + at(2, 1, 1));
            lane_of<K>(mu[3]) = at(0, 0, 1) + at(2, 0, 1);
            lane_of<K>(mu[4]) = at(0, -1, 1) + (at(2, -1, 1) - at(1, -1, 1));
            lane_of<K>(mu[5]) = at(0, -1, 0) - at(1, -1, 0);
            lane_of<K>(mu[6]) = at(0, -1, -1) - (at(1, -1, -1) + at(2, -1, -1));
            lane_of<K>(mu[7]) = at(0, 0, -1) - at(2, 0, -1);
            lane_of<K>(mu[8]) = at(0, 1, -1) + (at(1, 1, -1) - at(2, 1, -1));
        } else {
            const int x = ring_index(x0 + cc, nx), y = ring_index(y0 + rr, ny);
            const int xm = x == 0 ? nx - 1 : x - 1, xp = x + 1 == nx ? 0 : x + 1;
            const int r0 = y * nx, rD = (y == 0 ? ny - 1 : y - 1) * nx, rU = (y + 1 == ny ? 0 : y + 1) * nx;
            lane_of<K>(mu[0]) = ldro(an + in_plane(r0 + x));
            lane_of<K>(mu[1]) = ldro(an + (n + in_plane(r0 + xp)));
            lane_of<K>(mu[2]) = ldro(an + (2 * n + in_plane(rU + xp)));
            lane_of<K>(mu[3]) = ldro(an + (3 * n + in_plane(rU + x)));
            lane_of<K>(mu[4]) = ldro(an + (4 * n + in_plane(rU + xm)));
            lane_of<K>(mu[5]) = ldro(an + (5 * n + in_plane(r0 + xm)));
            lane_of<K>(mu[6]) = ldro(an + (6 * n + in_plane(rD + xm)));
            lane_of<K>(mu[7]) = ldro(an + (7 * n + in_plane(rD + x)));
            lane_of<K>(mu[8]) = ldro(an + (8 * n + in_plane(rD + xp)));
        }
    };
    const X third = pk(S(1.0 / 3.0)), twelfth = pk(S(1.0 / 12.0));
    // aF = sum_l 3 w_l c_l mu_l
    auto source = [&](const X(&mu)[9], X& aFx, X& aFy) {
        const X d26 = mu[2] - mu[6], d48 = mu[4] - mu[8];
        aFx = pfma(mu[1] - mu[5], third, (d26 - d48) * twelfth);
        aFy = pfma(mu[3] - mu[7], third, (d26 + d48) * twelfth);
    };
    X mu[9], aFx, aFy, ah, ajx, ajy;
    const X h = dh + pk(C.href);
    lanes([&](auto k_c) {
        constexpr int K = decltype(k_c)::value;
        gather(k_c, c, r + K * HALF, mu);
    });
    source(mu, aFx, aFy);
    {
        // adjoints through the equilibria (Eq. equilibria, e = 1) and the
        // source, summed over l in closed form; times omega
        const X ih = prcp(h), ux = jx * ih, uy = jy * ih, q = pfma(ux, ux, uy * uy), gh = pk(C.g) * h;
        const X p15 = mu[1] + mu[5], p37 = mu[3] + mu[7], p26 = mu[2] + mu[6], p48 = mu[4] + mu[8];
        const X sax = p15 + p37, sdg = p26 + p48, ua = ux + uy, ub = ux - uy;
        const X e1 = pfma(q, pk(S(2.0 / 3.0)), pfma(gh, pk(S(-5.0 / 3.0)), pk(S(1))));
        const X e2 = pfma(gh, third, q * pk(S(1.0 / 6.0)));
        const X squares = pfma(ux * ux, p15, uy * uy * p37), diags = pfma(ua * ua, p26, ub * ub * p48);
        ah = pfma(mu[0], e1, pfma(e2, pfma(sdg, pk(S(0.25)), sax), pfma(squares, pk(S(-0.5)), diags * pk(S(-0.125)))));
        const X lin = pfma(mu[0], pk(S(-4.0 / 3.0)), pneg(pfma(sax, third, sdg * twelfth)));
        const X ca = ua * p26, cb = ub * p48;
        ajx = pfma(ux, lin + p15, pfma(ca + cb, pk(S(0.25)), aFx));
        ajy = pfma(uy, lin + p37, pfma(ca - cb, pk(S(0.25)), aFy));
    }
    X agx = pneg(h * aFx), agy = pneg(h * aFy);
    lanes([&](auto k_c) {
        constexpr int K = decltype(k_c)::value;
        gxs[r + K * HALF + 2][c + 2] = lane_of<K>(agx);
        gys[r + K * HALF + 2][c + 2] = lane_of<K>(agy);
    });
    if (t < HP) {
        X m[9], fx, fy;
        lanes([&](auto k_c) { gather(k_c, hc[decltype(k_c)::value], hr[decltype(k_c)::value], m); });
        source(m, fx, fy);
        hh = hh + pk(C.href);
        X gx = pneg(hh * fx), gy = pneg(hh * fy);
        lanes([&](auto k_c) {
            constexpr int K = decltype(k_c)::value;
            gxs[hr[K] + 2][hc[K] + 2] = lane_of<K>(gx);
            gys[hr[K] + 2][hc[K] + 2] = lane_of<K>(gy);
        });
    }
    __syncthreads();

    if (RESIDENT != 1024 && early) dependent_launch_next();
    // ---- 3
    // p and -gamma ap from the h and ag windows; ap(x) = sum_l 3 w_l c_l . ag(x - c_l)
    auto both = [&](const Win<X>& H, const Win<X>& gx, const Win<X>& gy, X k, X& p, X& l, X& ih) {
        p = node_pressure(H, k, disj, C, ih);
        const X axis = (gx.cL - gx.cR) + (gy.s0 - gy.n0);
        const X diag = ((gx.sL + gy.sL) + (gy.sR - gx.sR)) + ((gx.nL - gy.nL) - (gx.nR + gy.nR));
        l = pmul(pk(-C.gamma), pfma(axis, third, diag * twelfth));
    };
    X ihn;
    {
        Win<X> H, gx, gy;
        X p, l;
        lanes([&](auto k_c) {
            constexpr int K = decltype(k_c)::value;
            tile_window<K>(&hs[r + K * HALF + 2][c + 2], HW, H);
            tile_window<K>(&gxs[r + K * HALF + 2][c + 2], HW, gx);
            tile_window<K>(&gys[r + K * HALF + 2][c + 2], HW, gy);
        });
        both(H, gx, gy, kap, p, l, ihn);
        lanes([&](auto k_c) {
            constexpr int K = decltype(k_c)::value;
            ps[r + K * HALF + 1][c + 1] = lane_of<K>(p);
            ls[r + K * HALF + 1][c + 1] = lane_of<K>(l);
        });
        // d/dkappa of Pi does not vanish where kappa does: always accumulate
        X api = pk(C.pi_sgn) * l;
        const X q = pk(C.hstar) * ihn;
        X rn, rm;
        if (C.n_exp == 3 && C.m_exp == 2) {
            rm = q * q;
            rn = rm * q;
        } else {
            rn = pipow(q, C.n_exp);
            rm = pipow(q, C.m_exp);
        }
        ah = pmul(pk(C.omega), ah) + api * kap * (pk(S(C.m_exp)) * rm - pk(S(C.n_exp)) * rn) * ihn;
        X sum = gold + api * (rn - rm);
        lanes([&](auto k_c) {
            constexpr int K = decltype(k_c)::value;
            const int x = x0 + c, y = y0 + r + K * HALF;
            if (x < nx && y < ny) gk[in_plane(y * nx + x)] = lane_of<K>(sum);
        });
    }
    if (t < PP) {
        Win<X> H, gx, gy;
        X p, l, q;
        lanes([&](auto k_c) {
            constexpr int K = decltype(k_c)::value;
            tile_window<K>(&hs[pr[K] + 2][pc[K] + 2], HW, H);
            tile_window<K>(&gxs[pr[K] + 2][pc[K] + 2], HW, gx);
            tile_window<K>(&gys[pr[K] + 2][pc[K] + 2], HW, gy);
        });
        both(H, gx, gy, kh, p, l, q);
        lanes([&](auto k_c) {
            constexpr int K = decltype(k_c)::value;
            ps[pr[K] + 1][pc[K] + 1] = lane_of<K>(p);
            ls[pr[K] + 1][pc[K] + 1] = lane_of<K>(l);
        });
    }
    __syncthreads();

    if (RESIDENT == 1024 || !early) dependent_launch_next();
    // ---- 4
    Win<X> P, L;
    lanes([&](auto k_c) {
        constexpr int K = decltype(k_c)::value;
        tile_window<K>(&ps[r + K * HALF + 1][c + 1], PW, P);
        tile_window<K>(&ls[r + K * HALF + 1][c + 1], PW, L);
    });
    const X gpx = pfma(P.cR - P.cL, third, ((P.nR - P.nL) + (P.sR - P.sL)) * twelfth);
    const X gpy = pfma(P.n0 - P.s0, third, ((P.nR - P.sR) + (P.nL - P.sL)) * twelfth);
    // Eqs. (forcefric, alphafric): nu alpha u = fr j, fr = 6 nu / (2h^2 + 6 delta h + 3 delta^2)
    const X den = pfma(h, pfma(pk(S(2)), h, pk(S(6) * C.delta)), pk(S(3) * C.delta * C.delta));
    const X iden = prcp(den), fr = pk(C.nu6) * iden;
    const X mdfr = fr * pfma(pk(S(4)), h, pk(S(6) * C.delta)) * iden;  // -d fr / dh
    ah = ah + pfma(aFx, pk(C.gx) - gpx, pfma(aFy, pk(C.gy) - gpy, mdfr * pfma(aFx, jx, aFy * jy)));
    const X axis = (L.cL + L.cR) + (L.n0 + L.s0), diag = (L.nL + L.nR) + (L.sL + L.sR);
    ah = pfma(pfma(pk(S(4)), axis, pfma(pk(S(-20)), L.c0, diag)), pk(S(1.0 / 6.0)), ah);
    ajx = pmul(pk(C.omega), ajx) - fr * aFx;
    ajy = pmul(pk(C.omega), ajy) - fr * aFy;
    X o[9];
    if constexpr (OMEGA1) {
        o[0] = ah;
        o[1] = ajx;
        o[2] = ajy;
    } else {
        const X om = pk(S(1) - C.omega), s = ajx + ajy, d = ajy - ajx;
        o[0] = pfma(om, mu[0], ah);
        o[1] = pfma(om, mu[1], ah + ajx);
        o[2] = pfma(om, mu[2], ah + s);
        o[3] = pfma(om, mu[3], ah + ajy);
        o[4] = pfma(om, mu[4], ah + d);
        o[5] = pfma(om, mu[5], ah - ajx);
        o[6] = pfma(om, mu[6], ah - s);
        o[7] = pfma(om, mu[7], ah - ajy);
        o[8] = pfma(om, mu[8], ah - d);
    }
    lanes([&](auto k_c) {
        constexpr int K = decltype(k_c)::value;
        const int x = x0 + c, y = y0 + r + K * HALF;
        if (x >= nx || y >= ny) return;
        S* out = a + in_plane(y * nx + x);
#pragma unroll
        for (int l = 0; l < (OMEGA1 ? 3 : 9); ++l) out[l * n] = lane_of<K>(o[l]);
    });
}

template <typename S, int TX, int TY>
cudaError_t adjoint_tile_one(const S* mom, bool fresh, const S* an, S* a, S* gk, const S* kappa, const Geom& G, const Consts<S>& C,
                             cudaStream_t st)
{
    constexpr int NT = TX * TY / Lanes<typename TileX<S>::X>::N;
    const dim3 grid((G.nx + TX - 1) / TX, (G.ny + TY - 1) / TY);
    // When the next step's CTAs may be placed (see tile_one): after ag where tiles
    // number at most one an SM or fill nearly all slots once, else after p (us a
    // backward step, after p / after ag: 128^2 4.8 / 4.3, 300 x 200 5.8 / 5.1,
    // 384^2 6.8 / 6.5; 320^2 6.8 / 7.2, 400^2 9.7 / 10.1, 512^2 9.6 / 9.8, 1024^2
    // 32.2 / 32.8; with the record fetched after the wait, after p: 128^2 4.8, 300
    // x 200 5.6, 512^2 10.2, 1024^2 33.0).
    const long long tiles = (long long)grid.x * grid.y, sms = sm_count(), slots = 512 / NT * sms;
    const bool early = tiles <= sms || (tiles <= slots && 6 * tiles >= 5 * slots);
    if (C.omega != S(1)) return launch_dependent(k_adjoint_tile<S, TX, TY, false, 512>, grid, NT, 0, st, mom, fresh, early, an, a, gk, kappa, G, C);
    // threads an SM holds, as for the forward tiles (one box, omega = 1, us of a
    // gradient a step with neither rule / both: 512^2 16.3 / 13.8, 768^2 29.7 / 25.6,
    // 1024^2 52.9 / 45.1; 384^2, below both, 9.1)
    if constexpr (TX == 32 && sizeof(S) == 4) {
        if (tiles > 3 * sms)
            return launch_dependent(k_adjoint_tile<S, TX, TY, true, 1024>, grid, NT, 0, st, mom, fresh, early, an, a, gk, kappa, G, C);
    }
    return launch_dependent(k_adjoint_tile<S, TX, TY, true, 512>, grid, NT, 0, st, mom, fresh, early, an, a, gk, kappa, G, C);
}

}  // namespace tflbm
