// Tile form of the fused step (Section II of Zitz et al., arXiv:1810.07642),
// for lattices that the L2 cache holds.
//
// Why: the marching kernels (tflbm_step.cuh, tflbm_step2.cuh) walk a band row
// by row, each row waiting for loads of the row before; a band of 16 rows is a
// chain of 21 L2 round trips and barriers, about 14 us whatever the lattice's
// size, and a small lattice has too few bands to hide them.  Here a CTA owns a
// tile of TX x TY nodes and runs the step's three phases over all of it: pull
// and moments of the tile and a halo of 2 (every load of the tile in flight at
// once), a barrier, the pressure of the tile and a halo of 1, a barrier, force
// and collision: one round trip and two barriers a step.  The halo costs
// repeated pulls (1.4 a node at 32 x 16), which come from L1/L2; on a lattice
// much larger than L2 the march, which pulls each node about 1.3 times and
// loads ahead, is the faster one.
//
// A thread owns X::N nodes of its tile (FP32 compute type: two, TY / 2 rows
// apart, on the paired FP32 instructions; FP64: one) and keeps their momenta
// (and, when omega != 1, their pulled populations) in registers between the
// phases; halo nodes only leave h or p in shared memory.  Columns and rows are
// wrapped per node, so any lattice down to one node works; nodes of a tile that
// lie past the lattice's edge are computed as their periodic images and not
// stored.  The node arithmetic is that of tflbm_node.cuh.
#pragma once
#include "tflbm_handle.h"
#include "tflbm_node.cuh"

namespace tflbm {

// i on a ring of n (the modulo only runs outside the lattice)
__device__ __forceinline__ int ring_index(int i, int n) { return (unsigned)i < (unsigned)n ? i : wrap_index(i, n); }

template <typename S> struct TileX { using X = float2; };
template <> struct TileX<double> { using X = double; };

// lane k of x
template <int K> __device__ __forceinline__ float& lane_of(float2& x)
{
    if constexpr (K == 0) return x.x;
    else return x.y;
}
template <int K> __device__ __forceinline__ double& lane_of(double& x) { return x; }

// Position of node i of the halo of depth D around a TX x TY tile: D rows
// below and above over the whole width, then the columns on both sides.
template <int TX, int TY, int D>
__device__ __forceinline__ void tile_halo(int i, int& c, int& r)
{
    constexpr int W = TX + 2 * D;
    if (i < 2 * D * W) {
        const int k = i / W;
        c = i % W - D;
        r = k < D ? k - D : TY + k - D;
    } else {
        const int k = (i - 2 * D * W) % (2 * D);
        r = (i - 2 * D * W) / (2 * D);
        c = k < D ? k - D : TX + k - D;
    }
}

// Lane K of the window around element b of rows w wide.
template <int K, typename S, typename X>
__device__ __forceinline__ void tile_window(const S* b, int w, Win<X>& W)
{
    lane_of<K>(W.nL) = b[w - 1]; lane_of<K>(W.n0) = b[w]; lane_of<K>(W.nR) = b[w + 1];
    lane_of<K>(W.cL) = b[-1]; lane_of<K>(W.c0) = b[0]; lane_of<K>(W.cR) = b[1];
    lane_of<K>(W.sL) = b[-w - 1]; lane_of<K>(W.s0) = b[-w]; lane_of<K>(W.sR) = b[-w + 1];
}

// Moments of the nine pulled populations n (storage units).
template <typename SM, typename X>
__device__ __forceinline__ void node_moments(X f0, const X (&n)[8], const Consts<typename Lanes<X>::S>& C, X& dh, X& er,
                                             X& jx, X& jy)
{
    const X Rs = padd(n[0], padd(n[1], n[7])), Ls = padd(n[4], padd(n[3], n[5]));
    const X jyr = padd(psub(n[2], n[6]), padd(psub(n[1], n[7]), psub(n[3], n[5])));
    node_moments<SM>(f0, Rs, Ls, padd(n[2], n[6]), jyr, C, dh, er, jx, jy);
}

template <typename SM, typename S, int TX, int TY, bool OMEGA1, int RESIDENT>
__global__ void __launch_bounds__(TX* TY / Lanes<typename TileX<S>::X>::N, RESIDENT / (TX * TY / Lanes<typename TileX<S>::X>::N))
k_tile(const S* __restrict__ fin0, const SM* __restrict__ finm, S* __restrict__ fout0, SM* __restrict__ foutm,
       const S* __restrict__ kappa, S* __restrict__ mom, bool early, const Geom G, const Consts<S> C)
{
    using X = typename TileX<S>::X;
    using IO = PairIO<SM>;
    using V = typename IO::V;
    constexpr int N = Lanes<X>::N, NT = TX * TY / N, HALF = TY / N;
    constexpr int HW = TX + 4, PW = TX + 2;
    // halo nodes of the h and p rings around the tile, and pairs of them
    constexpr int HN = HW * (TY + 4) - TX * TY, PN = PW * (TY + 2) - TX * TY;
    constexpr int HP = HN / N, PP = PN / N;
    static_assert(HN % N == 0 && PN % N == 0 && TY % N == 0, "halo nodes come in whole groups");
    static_assert(HP <= NT && PP <= NT, "one group of halo nodes a thread");
    __shared__ S hs[TY + 4][HW];  // h - href; tile node (c, r) at [r + 2][c + 2]
    __shared__ S ps[TY + 2][PW];  // p; tile node (c, r) at [r + 1][c + 1]

    const int t = threadIdx.x, nx = G.nx, ny = G.ny, pitch = G.pitch, plane = (int)G.plane;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int c = t % TX, r = t / TX;  // own nodes: (c, r + k HALF)
    const bool disj = kappa != nullptr || C.kappa_u != S(0);

    // where the populations arriving at a node lie: its columns x - 1, x, x + 1
    // and the offsets of its rows y - 1, y, y + 1
    struct Spot {
        uint32_t xm, x, xp, rm, r0, rp;
    };
    auto spot = [&](int cc, int rr) -> Spot {
        const int x = ring_index(x0 + cc, nx), y = ring_index(y0 + rr, ny);
        return {(uint32_t)(x == 0 ? nx - 1 : x - 1), (uint32_t)x, (uint32_t)(x + 1 == nx ? 0 : x + 1),
                (uint32_t)((y == 0 ? ny - 1 : y - 1) * pitch), (uint32_t)(y * pitch),
                (uint32_t)((y + 1 == ny ? 0 : y + 1) * pitch)};
    };
    // load them into lane K: a uniform plane and a 32-bit offset within it, one
    // register an access
    auto pull = [&](auto k_c, const Spot& p, X& f0, X (&n)[8]) {
        constexpr int K = decltype(k_c)::value;
        int* st = C.status;
        (void)st;
        auto at = [&](int l, uint32_t i) { return IO::dec1(ldro(finm + l * plane + TFLBM_IDX(i, plane, st))); };
        lane_of<K>(f0) = ldro(fin0 + TFLBM_IDX(p.r0 + p.x, plane, st));
        lane_of<K>(n[0]) = at(0, p.r0 + p.xm);
        lane_of<K>(n[1]) = at(1, p.rm + p.xm);
        lane_of<K>(n[2]) = at(2, p.rm + p.x);
        lane_of<K>(n[3]) = at(3, p.rm + p.xp);
        lane_of<K>(n[4]) = at(4, p.r0 + p.xp);
        lane_of<K>(n[5]) = at(5, p.rp + p.xp);
        lane_of<K>(n[6]) = at(6, p.rp + p.x);
        lane_of<K>(n[7]) = at(7, p.rp + p.xm);
    };
    auto kap_at = [&](int cc, int rr) -> S {
        if (!kappa) return C.kappa_u;
        const long long nk = (long long)nx * ny;
        (void)nk;
        return ldro(kappa + TFLBM_IDX(ring_index(y0 + rr, ny) * nx + ring_index(x0 + cc, nx), nk, C.status));
    };
    auto lanes = [&](auto fn) {
        fn(std::integral_constant<int, 0>{});
        if constexpr (N == 2) fn(std::integral_constant<int, 1>{});
    };

    // ---- before the previous step has ended: places, and kappa (which it does
    // not write)
    X f0, n[8], dh, er, jx, jy, kap, kh, ih;
    Spot own[N], beside[N];
    int hc[N], hr[N], pc[N], pr[N];
    lanes([&](auto k_c) {
        constexpr int K = decltype(k_c)::value;
        own[K] = spot(c, r + K * HALF);
        lane_of<K>(kap) = kap_at(c, r + K * HALF);
        if (t < HP) {
            tile_halo<TX, TY, 2>(t + K * HP, hc[K], hr[K]);
            beside[K] = spot(hc[K], hr[K]);
        }
        if (t < PP) {
            tile_halo<TX, TY, 1>(t + K * PP, pc[K], pr[K]);
            lane_of<K>(kh) = kap_at(pc[K], pr[K]);
        }
    });
    dependent_launch_wait();
    // ---- h and j of the tile, h of the halo of 2
    lanes([&](auto k_c) { pull(k_c, own[decltype(k_c)::value], f0, n); });
    if (t < HP) {
        X g0, g[8], d, e, a, b;
        lanes([&](auto k_c) { pull(k_c, beside[decltype(k_c)::value], g0, g); });
        node_moments<SM>(g0, g, C, d, e, a, b);
        lanes([&](auto k_c) {
            constexpr int K = decltype(k_c)::value;
            hs[hr[K] + 2][hc[K] + 2] = lane_of<K>(d);
        });
    }
    node_moments<SM>(f0, n, C, dh, er, jx, jy);
    lanes([&](auto k_c) {
        constexpr int K = decltype(k_c)::value;
        hs[r + K * HALF + 2][c + 2] = lane_of<K>(dh);
        const int x = x0 + c, y = y0 + r + K * HALF;
        if (mom && x < nx && y < ny) {
            const long long nn = (long long)nx * ny;
            S* m = mom + (y * nx + x);
            m[0] = lane_of<K>(dh);
            m[nn] = lane_of<K>(jx);
            m[2 * nn] = lane_of<K>(jy);
        }
    });
    __syncthreads();

    if (early) dependent_launch_next();
    // ---- film pressure of the tile and the halo of 1
    {
        Win<X> W;
        lanes([&](auto k_c) {
            constexpr int K = decltype(k_c)::value;
            tile_window<K>(&hs[r + K * HALF + 2][c + 2], HW, W);
        });
        X p = node_pressure(W, kap, disj, C, ih);
        lanes([&](auto k_c) {
            constexpr int K = decltype(k_c)::value;
            ps[r + K * HALF + 1][c + 1] = lane_of<K>(p);
        });
    }
    if (t < PP) {
        Win<X> W;
        X q;
        lanes([&](auto k_c) {
            constexpr int K = decltype(k_c)::value;
            tile_window<K>(&hs[pr[K] + 2][pc[K] + 2], HW, W);
        });
        X p = node_pressure(W, kh, disj, C, q);
        lanes([&](auto k_c) {
            constexpr int K = decltype(k_c)::value;
            ps[pr[K] + 1][pc[K] + 1] = lane_of<K>(p);
        });
    }
    __syncthreads();

    if (!early) dependent_launch_next();
    // ---- force, collision and store of the tile
    Win<X> W;
    lanes([&](auto k_c) {
        constexpr int K = decltype(k_c)::value;
        tile_window<K>(&ps[r + K * HALF + 1][c + 1], PW, W);
    });
    node_collide<SM, OMEGA1>(W, dh, ih, jx, jy, er, n, 1, C, [&](X o0, const V(&q)[8]) {
        const int x = x0 + c;
        lanes([&](auto k_c) {
            constexpr int K = decltype(k_c)::value;
            const int y = y0 + r + K * HALF;
            if (x >= nx || y >= ny) return;
            const uint32_t i = TFLBM_IDX((uint32_t)(y * pitch + x), plane, C.status);
            fout0[i] = lane_of<K>(o0);
#pragma unroll
            for (int l = 0; l < 8; ++l) {
                SM v;
                if constexpr (N == 1) v = q[l];
                else if constexpr (K == 0) v = q[l].x;
                else v = q[l].y;
                (foutm + l * plane)[i] = v;
            }
        });
    });
}

template <typename SM, typename S, int TX, int TY>
cudaError_t tile_one(const S* f0, const SM* fm, S* g0, SM* gm, const S* kappa, S* mom, const Geom& G,
                     const Consts<S>& C, cudaStream_t st)
{
    constexpr int NT = TX * TY / Lanes<typename TileX<S>::X>::N;
    const dim3 grid((G.nx + TX - 1) / TX, (G.ny + TY - 1) / TY);
    // When the next step's CTAs may be placed.  As soon as this step starts, they
    // go to the SMs that have room then, two or three to one and none to another
    // (us a step against after the pressure: FP64 tau = 0.8 128^2 25.3 / 8.5, 250
    // x 190 25.2 / 20.1).  After the pressure, every tile is on an SM and near
    // its end; after h already, another phase of the next step's preamble and
    // launch is hidden, but the placement is uneven again unless half of the SMs
    // are empty, small tiles number at most one an SM, or at least 5/6 of the
    // slots are full (one wave, or several: the sizes measured have up to 13.5
    // tiles an SM).  FP32, us a step, after the pressure / after
    // h: 64^2 2.61 / 2.45, 128^2 2.77 / 2.55, 200 x 150 (130 tiles of 16 x 16) 3.22
    // / 2.90; 256^2 (128 of 32 x 16) 3.03 / 3.18, 320^2 (400 of 16 x 16) 3.41 /
    // 3.67, 384^2 (288 of 32 x 16) 3.54 / 3.83; 509 x 387 (400) 4.58 / 4.23, 512^2
    // (512) 4.70 / 4.58, 1024^2 14.95 / 14.80.  With records 512^2 loses 0.08.
    // Without a kappa field the preamble is too short to hide anything (one kappa,
    // 128^2 2.32 / 2.51, 512^2 4.45 / 4.51).
    const long long tiles = (long long)grid.x * grid.y, sms = sm_count();
    const long long slots = (tiles > 3 * sms ? 4 : 3) * sms;  // of FP32 32 x 16 tiles, see below
    const bool spread = 2 * tiles <= sms || (TX * TY <= 256 && tiles <= sms) ||
                       (TX == 32 && sizeof(S) == 4 && !mom && 6 * tiles >= 5 * slots);
    const bool early = kappa && spread;
    auto launch = [&](auto resident) {
        constexpr int R = decltype(resident)::value;
        if (C.omega == S(1)) return launch_dependent(k_tile<SM, S, TX, TY, true, R>, grid, NT, 0, st, f0, fm, g0, gm, kappa, mom, early, G, C);
        return launch_dependent(k_tile<SM, S, TX, TY, false, R>, grid, NT, 0, st, f0, fm, g0, gm, kappa, mom, early, G, C);
    };
    // Threads an SM holds.  768 leaves the registers that keep a thread's 18
    // loads in flight (80); where 32 x 16 tiles outnumber the three an SM
    // holds then, 64 registers and a fourth tile win (one box, tau = 1, us a step
    // with 768 / 1024: 512^2 6.12 / 4.53, 640 x 480 6.36 / 4.57, 768^2 10.2 / 8.7, 1024^2
    // 18.0 / 15.1; 509 x 387, 2.6 tiles an SM, 4.24 with 768).
    if constexpr (TX == 32 && sizeof(S) == 4) {
        if (tiles > 3 * sms) return launch(std::integral_constant<int, 1024>{});
    }
    return launch(std::integral_constant<int, sizeof(S) == 4 ? 768 : 512>{});
}

// One step from fin to fout in the tiles that block_x names (tile_of); mom, if
// not null, receives (h - href, j_x, j_y) of the state that fin pulls to,
// [3][ny][nx] (the gradient tape's record of the step).
template <typename SM, typename S>
cudaError_t tile_step(int block_x, const void* fin, void* fout, const void* kappa, void* mom, const Geom& G,
                      const Consts<S>& C, cudaStream_t st)
{
    const S* f0 = (const S*)fin;
    const SM* fm = (const SM*)((const char*)fin + G.plane * sizeof(S));
    S* g0 = (S*)fout;
    SM* gm = (SM*)((char*)fout + G.plane * sizeof(S));
    const S* k = (const S*)kappa;
    S* m = (S*)mom;
    switch (block_x) {
        case 64: return tile_one<SM, S, 16, 8>(f0, fm, g0, gm, k, m, G, C, st);
        case 128: return tile_one<SM, S, 16, 16>(f0, fm, g0, gm, k, m, G, C, st);
        case 256: return tile_one<SM, S, 32, 16>(f0, fm, g0, gm, k, m, G, C, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace tflbm
