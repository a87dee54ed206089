// Four-column march: the fused step (Section II of Zitz et al.,
// arXiv:1810.07642) at omega = 1 with an FP32 compute type, forcing = 0, for
// lattices larger than L2.
//
// What bounds it, and what it does about it.  At 2048^2 the two-column march
// (tflbm_step2.cuh) moved 76 B a node at 0.9 of the copy bandwidth in FP32 and
// was bound by instruction issue with 16-bit populations.
//  * Moments between steps (FP32).  At omega = 1 the post-collision populations
//    of a node are a function of six numbers: h - href, the residual of its
//    sum, the momentum j and G = j + F (the even parts of f* come from h and
//    j/h, the odd parts from G, the rest population from both).  Between two
//    steps of one call the kernel keeps those six planes, 24 B a node and
//    direction in place of 36, and the next step forms the nine populations
//    from them with the instructions that would have stored them.  The first
//    step of a call reads populations and the last one writes them, so what a
//    call leaves behind is the population buffer, with the same bits whatever
//    the number of steps per call.
//  * Four columns a thread, one warp a CTA (128 columns).  The values that
//    cross a thread's columns take four shuffles a row, the stencils' outer
//    neighbours two each for h and p; every row of h and p that a stencil needs
//    stays in registers, so a row has no barrier and no shared-memory exchange.
//    What a thread needs of its own columns two rows later (j and the residual
//    of the sum) waits in its own slots of a shared ring.
// 2048^2, us a step, two-column march and this one: FP32 53.5 / 39.4 (52 B and
// 19.5 M warp instructions a step against 76 B and 32.1 M), FP16 44.3 / 37.0;
// 1448^2 FP32 40.2 / 21.7; 2047 x 2049 FP32 (one column) 60 / 44.5.  What is left:
// twelve warps an SM issue half of the slots (long-scoreboard and fixed-latency
// stalls), HBM 55 % busy.
//
// Streaming.  A thread holds f* of row r(k) at its own columns (loaded, or
// formed from the moments).  Its populations with c_y = +1 belong to row r(k+1),
// those with c_y = -1 to row r(k-1), the others to r(k); each row's sums are
// complete one row later.  The march mirrors the lattice when it runs towards
// -y (j_y, G_y and g_y change sign, populations 2, 3, 4 exchange with 8, 7, 6):
// every sum of the node arithmetic (tflbm_node.cuh) gives the same bits then.
//
// Iteration k: f* of row r(k) (copies of row r(k+2) requested); h, j of row
// r(k-1); pressure of row r(k-2); force, collision and store of row r(k-3).
// Local columns 0 .. 127 are x0 - 4 .. x0 + 123, x0 a multiple of 4; h is right
// on 1 .. 126, p on 2 .. 125, the output is 4 .. 123 (120 columns): every access
// of a thread is one aligned group of four columns.  (122 output columns in
// pairs of columns instead: twice the accesses, L1's data stage 68 % busy, 43.6
// us a 2048^2 FP32 step.)  QUAD: nx is a multiple of 4, groups wrap whole and the
// code has no branch on the columns (with one, 48 us).  Otherwise a moments row
// carries the four columns beyond either end as well, so that its groups never
// wrap, and a population row's groups that wrap load one by one.
#pragma once
#include "tflbm_tile.cuh"

namespace tflbm {

constexpr int kWideCols = 120;  // output columns of a strip

// Planes of a moments buffer.
enum { kMomH = 0, kMomE, kMomJx, kMomJy, kMomGx, kMomGy, kMomPlanes };
// Elements of a moments row: columns -4 .. nx + 3 at 0 .. nx + 7, padded to a
// whole number of groups.  A strip's window may run up to 124 elements past its
// row; wide_applies says whether the planes, with that, fit a population buffer.
__host__ __device__ inline int mom_pitch(int nx) { return (nx + 8 + 3) / 4 * 4; }

// One row of h or p at the thread's columns (NP pairs) and the two beside them.
constexpr int NP = 2;
struct WideRow {
    float2 c[NP];
    float l, r;
    // fill in the columns beside from the neighbouring lanes
    __device__ __forceinline__ void sides()
    {
        l = __shfl_up_sync(0xffffffffu, c[NP - 1].y, 1);
        r = __shfl_down_sync(0xffffffffu, c[0].x, 1);
    }
    // pair p shifted one column to the left (its nodes' left neighbours) and to the right
    __device__ __forceinline__ float2 left(int p) const { return make_float2(p == 0 ? l : c[p - 1].y, c[p].x); }
    __device__ __forceinline__ float2 right(int p) const { return make_float2(c[p].y, p == NP - 1 ? r : c[p + 1].x); }
};
// the window of the thread's pair p
__device__ __forceinline__ Win<float2> wide_window(const WideRow& n, const WideRow& c, const WideRow& s, int p)
{
    return {n.c[p], n.left(p), n.right(p), c.c[p], c.left(p), c.right(p), s.c[p], s.left(p), s.right(p)};
}
// a thread's four consecutive values
__device__ __forceinline__ void lds_pairs(const float* p, float2 (&v)[NP])
{
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = make_float2(q.x, q.y);
    v[1] = make_float2(q.z, q.w);
}
__device__ __forceinline__ void sts_pairs(float* p, const float2 (&v)[NP])
{
    *reinterpret_cast<float4*>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
}

// Four elements, 16 (or, of a 16-bit type, 8) bytes; .cg: through L2 only.
template <typename E>
__device__ __forceinline__ void cp_async4(E* dst, const E* src)
{
    if constexpr (sizeof(E) == 4)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
    else
        cp_async<8>(dst, src);
}

// MOM_IN / MOM_OUT: the source / the destination holds moments (SM = float).
template <typename SM, bool MOM_IN, bool MOM_OUT, bool QUAD>
__device__ __forceinline__ void step_band4(const void* __restrict__ fin, void* __restrict__ fout,
                                           const float* __restrict__ kappa, const Geom& G, const Consts<float>& C0,
                                           int strip, int band, int nbands)
{
    static_assert((!(MOM_IN || MOM_OUT) && QUAD) || sizeof(SM) == 4, "moments and ragged rows go with FP32 storage");
    using IO = PairIO<SM>;
    using V = typename IO::V;
    // rows on their way: full-width planes, and 8 moving planes of the storage type
    constexpr int kAhead = sizeof(SM) == 4 && !MOM_IN ? 1 : 2, kStagesW = kAhead + 1;
    constexpr int kFull = MOM_IN ? (int)kMomPlanes : 1;
    constexpr int NC = 128;
    __shared__ __align__(16) float wide[kStagesW][kFull][NC];
    __shared__ __align__(16) SM moving[MOM_IN ? 1 : kStagesW][MOM_IN ? 1 : 8][MOM_IN ? 8 : NC];
    // the thread's j_x, j_y and sum residual of the last three rows
    __shared__ __align__(16) float ring[3][3][NC];

    const int t = threadIdx.x;
    const int nx = G.nx, ny = G.ny, pitch = G.pitch, plane = (int)G.plane;
    const int x0 = strip * kWideCols, weff = min(kWideCols, nx - x0);
    const int ybeg = (int)(((long long)band * ny) / nbands), yend = (int)(((long long)(band + 1) * ny) / nbands);
    const int dir = ((band + C0.flip) & 1) ? -1 : 1;  // reversed every other step (see make_band)
    const int R = yend - ybeg;
    const float sgn = (float)dir;
    Consts<float> C = C0;
    C.gy *= sgn;
    C.forcing = 0;
    const bool disj = kappa != nullptr || C.kappa_u != 0.0f;

    // the thread's columns: xt .. xt + 3; its share of the output
    const int xt = x0 - 4 + 4 * t, xw = wrap_index(xt, nx);
    const bool inside = QUAD || (xt >= 0 && xt + 3 < nx);   // an aligned group of a population row
    const bool whole = t >= 1 && 4 * t <= weff, part = !QUAD && t >= 1 && !whole && 4 * t < weff + 4;
    // this strip writes columns that the row's ends repeat
    const bool ends = !QUAD && (x0 == 0 || x0 + weff > nx - 4);
    const int mpitch = QUAD ? pitch : mom_pitch(nx), mplane = ny * mpitch;
    const int xg = QUAD ? xw : xt, xm = QUAD ? xw : xt + 4;  // the group in a population and in a moments row
    (void)mplane;
    // offsets within a moments plane at which the last plane's group still lies in
    // the population buffer
    const long long mroom = 9LL * plane - (kMomPlanes - 1LL) * mplane - 3;
    (void)mroom;
    TFLBM_CHECK(!whole || (xm >= 0 && xm + 3 < mpitch && xg >= 0 && xg + 3 < nx), C.status);
    const float* __restrict__ in0 = (const float*)fin;
    const SM* __restrict__ inm = (const SM*)(in0 + plane);
    float* __restrict__ out0 = (float*)fout;
    SM* __restrict__ outm = (SM*)(out0 + plane);
    const long long nk = (long long)nx * ny;
    (void)nk;
    // plane (l - 1) of population l in the mirrored frame
    auto plane_of = [&](int l) { return l == 0 || l == 4 || dir > 0 ? l : 8 - l; };
    // Offsets within a plane are 32-bit, so that an access is a uniform base and
    // one register.
    auto store_group = [&](auto* __restrict__ base, uint32_t off, const auto (&v)[NP]) {  // off: the group's
        using P2 = typename std::remove_const<typename std::remove_reference<decltype(v[0])>::type>::type;
        using P4 = typename std::conditional<sizeof(P2) == 8, float4, uint2>::type;
        if (whole) {  // predicated stores
            P4 q;
            memcpy(&q, &v[0], sizeof(P2));
            memcpy((char*)&q + sizeof(P2), &v[1], sizeof(P2));
            *reinterpret_cast<P4*>(base + off) = q;
        }
    };
    // the columns of a group that store_group leaves out: the last ones of an
    // nx that is no multiple of 4, and in a moments row the images beyond the
    // ends (only in strips with odd: one branch a row)
    const bool odd = !QUAD && (ends || weff % 4 != 0);
    auto store_odd = [&](auto* __restrict__ row, bool images, const auto (&v)[NP]) {  // row: at column 0
        TFLBM_CHECK(!part || (xt >= 0 && xt < nx), C.status);
        if (part) {
            row[xt] = v[0].x;
            if (xt + 1 < nx) row[xt + 1] = v[0].y;
            if (xt + 2 < nx) row[xt + 2] = v[1].x;
        }
        if (images && ends && (whole || part)) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int x = xt + i;
                const auto c = i == 0 ? v[0].x : (i == 1 ? v[0].y : (i == 2 ? v[1].x : v[1].y));
                TFLBM_CHECK(x >= 0 && nx >= 4 && nx + 8 <= mpitch, C.status);
                if (x < 4) row[nx + x] = c;
                if (x >= nx - 4 && x < nx) row[x - nx] = c;
            }
        }
    };

    // The source rows in flight: each thread copies its own columns of
    // every plane into its own slots of a stage, kAhead rows before it reads
    // them.  (Prefetched into registers instead, the loads sank to their uses
    // under register pressure: 73 us a 2048^2 FP32 step in place of 52; three
    // rows ahead in place of two: 40.0 in place of 39.8.)
    auto copy = [&](auto* dst, const auto* __restrict__ row, bool groups) {  // dst: 4 elements; row: of a population plane
        using E = typename std::remove_reference<decltype(*dst)>::type;
        if (groups) {
            cp_async4<E>(dst, row + TFLBM_IDX(xg, pitch - 3, C.status));
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if constexpr (!QUAD) cp_async<sizeof(E)>(dst + i, row + wrap_index(xt + i, nx));
            }
        }
    };
    const bool groups = QUAD || __all_sync(0xffffffffu, inside);
    auto copy_row = [&](int st, int y) {
        TFLBM_CHECK(y >= 0 && y < ny, C.status);
        if constexpr (MOM_IN) {
            // the window may run past its row (see mom_pitch), not past the buffer
            const uint32_t off = TFLBM_IDX((uint32_t)y * (uint32_t)mpitch + (uint32_t)xm, mroom, C.status);
#pragma unroll
            for (int f = 0; f < kMomPlanes; ++f) cp_async4<float>(&wide[st][f][4 * t], in0 + f * mplane + off);
        } else {
            auto all = [&](bool g) {
                copy(&wide[st][0][4 * t], in0 + y * pitch, g);
#pragma unroll
                for (int l = 0; l < 8; ++l) copy(&moving[st][l][4 * t], inm + plane_of(l) * plane + y * pitch, g);
            };
            if (groups) all(true);
            else all(false);
        }
        cp_async_commit();
    };
    // populations l = 2, 3, 4 of the last two rows, f_0, l = 1 and 5 of the last
    float2 E1[3][NP], E2[3][NP], W[3][NP];
    WideRow H[3], P[3];
    float2 ih[3][NP], kap[NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            E1[i][p] = E2[i][p] = W[i][p] = ih[i][p] = H[i].c[p] = P[i].c[p] = pk(0.0f);
            H[i].l = H[i].r = P[i].l = P[i].r = 0.0f;
        }
        kap[p] = pk(C.kappa_u);
    }

    const int rstart = dir > 0 ? ybeg - 3 : yend + 2;
    int wn = wrap_index(rstart, ny);  // the next row to copy
    int wk = wrap_index(rstart - dir, ny);  // row r(k-1), whose kappa is loaded at iteration k
    auto adv = [&](int& w) {
        w += dir;
        w = w == ny ? 0 : (w < 0 ? ny - 1 : w);
    };
    const int last = R + 5;
    for (int i = 0; i < kAhead; ++i) {
        copy_row(i, wn);
        adv(wn);
    }
    int st = 0, stn = kAhead;  // stages of rows r(k) and r(k + kAhead)
    auto body = [&](auto s_c, int k) {
        constexpr int s = decltype(s_c)::value;          // slot of rows r(k-1) of h, r(k-2) of p
        constexpr int sp = (s + 2) % 3, spp = (s + 1) % 3;  // one and two rows before
        // ---- f* of row r(k) at the own columns, storage units
        cp_async_wait<kAhead - 1>();
        float2 f0[NP], o[NP][8], m[kFull][NP];
#pragma unroll
        for (int f = 0; f < kFull; ++f) lds_pairs(&wide[st][f][2 * NP * t], m[f]);
        if constexpr (!MOM_IN) {
#pragma unroll
            for (int l = 0; l < 8; ++l) {
                const SM* src = &moving[st][l][2 * NP * t];
#pragma unroll
                for (int p = 0; p < NP; ++p) o[p][l] = IO::dec(reinterpret_cast<const V*>(src)[p]);
            }
        }
        // rows beyond the last are not read; an empty group keeps the count
        if (k + kAhead <= last) {
            copy_row(stn, wn);
            adv(wn);
        } else {
            cp_async_commit();
        }
        st = st + 1 == kStagesW ? 0 : st + 1;
        stn = stn + 1 == kStagesW ? 0 : stn + 1;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            if constexpr (MOM_IN) {
                const float2 dh = m[kMomH][p], jx = m[kMomJx][p], Gx = m[kMomGx][p];
                const float2 jy = pmul(m[kMomJy][p], pk(sgn)), Gy = pmul(m[kMomGy][p], pk(sgn));
                const float2 h = padd(dh, pk(C.href)), i1 = prcp(h), ux = pmul(jx, i1), uy = pmul(jy, i1);
                float2 Sx, Sy, Sa, Sb;
                node_even<SM>(h, ux, uy, jx, jy, C, Sx, Sy, Sa, Sb);
                node_odd<SM>(Sx, Sy, Sa, Sb, Gx, Gy, C, o[p]);
                f0[p] = node_fold(dh, m[kMomE][p], o[p]);
            } else {
                f0[p] = m[0][p];
            }
        }
        float2 kap2[NP];  // kappa of row r(k-2)
#pragma unroll
        for (int p = 0; p < NP; ++p) kap2[p] = kap[p];
        if (kappa) {
            const float* row = kappa + TFLBM_IDX(wk * nx, nk, C.status);
            if constexpr (QUAD) {
                TFLBM_CHECK(xw >= 0 && xw + 3 < nx, C.status);
                lds_pairs(row + xw, kap);
            } else {
                const int x1 = xw + 1 == nx ? 0 : xw + 1, x2 = x1 + 1 == nx ? 0 : x1 + 1, x3 = x2 + 1 == nx ? 0 : x2 + 1;
                kap[0] = make_float2(__ldg(row + xw), __ldg(row + x1));
                kap[1] = make_float2(__ldg(row + x2), __ldg(row + x3));
            }
        }
        adv(wk);
        // ---- h and j of row r(k-1)
        float2 Pc[NP], Py[NP], Qc[NP], Qy[NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            Pc[p] = padd(W[1][p], padd(E2[0][p], o[p][7]));
            Py[p] = psub(E2[0][p], o[p][7]);
            Qc[p] = padd(W[2][p], padd(E2[2][p], o[p][5]));
            Qy[p] = psub(E2[2][p], o[p][5]);
        }
        const float pl = __shfl_up_sync(0xffffffffu, Pc[NP - 1].y, 1), pyl = __shfl_up_sync(0xffffffffu, Py[NP - 1].y, 1);
        const float qr = __shfl_down_sync(0xffffffffu, Qc[0].x, 1), qyr = __shfl_down_sync(0xffffffffu, Qy[0].x, 1);
        float2 er[NP], jx[NP], jy[NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const float2 Rs = make_float2(p == 0 ? pl : Pc[p - 1].y, Pc[p].x);
            const float2 Ry = make_float2(p == 0 ? pyl : Py[p - 1].y, Py[p].x);
            const float2 Ls = make_float2(Qc[p].y, p == NP - 1 ? qr : Qc[p + 1].x);
            const float2 Ly = make_float2(Qy[p].y, p == NP - 1 ? qyr : Qy[p + 1].x);
            const float2 jyr = padd(psub(E2[1][p], o[p][6]), padd(Ry, Ly));
            node_moments<SM>(W[0][p], Rs, Ls, padd(E2[1][p], o[p][6]), jyr, C, H[s].c[p], er[p], jx[p], jy[p]);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                E2[i][p] = E1[i][p];
                E1[i][p] = o[p][i + 1];
            }
            W[0][p] = f0[p];
            W[1][p] = o[p][0];
            W[2][p] = o[p][4];
        }
        sts_pairs(&ring[s][0][2 * NP * t], jx);
        sts_pairs(&ring[s][1][2 * NP * t], jy);
        sts_pairs(&ring[s][2][2 * NP * t], er);
        H[s].sides();
        // ---- pressure of row r(k-2)
        if (k >= 4) {
#pragma unroll
            for (int p = 0; p < NP; ++p)
                P[s].c[p] = node_pressure(wide_window(H[s], H[sp], H[spp], p), kap2[p], disj, C, ih[s][p]);
            P[s].sides();
        }
        // ---- force, collision and store of row r(k-3)
        if (k >= 6) {
            const int y = rstart + (k - 3) * dir;  // inside [ybeg, yend), no wrap
            TFLBM_CHECK(y >= 0 && y < ny, C.status);
            float2 kx[NP], ky[NP], e[NP], Gx[NP], Gy[NP], r0[NP], n[8][NP];
            V v[8][NP];
            lds_pairs(&ring[spp][0][2 * NP * t], kx);
            lds_pairs(&ring[spp][1][2 * NP * t], ky);
            lds_pairs(&ring[spp][2][2 * NP * t], e);
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const float2 d = H[spp].c[p], h = padd(d, pk(C.href));
                float2 ux, uy, ex, ey, Fx, Fy;
                node_force(wide_window(P[s], P[sp], P[spp], p), h, ih[sp][p], kx[p], ky[p], C, ux, uy, ex, ey, Fx, Fy);
                Gx[p] = padd(ex, Fx);
                Gy[p] = padd(ey, Fy);
                if constexpr (MOM_OUT) {
                    ky[p] = pmul(ky[p], pk(sgn));
                    Gy[p] = pmul(Gy[p], pk(sgn));
                } else {
                    float2 Sx, Sy, Sa, Sb, q[8];
                    node_even<SM>(h, ux, uy, ex, ey, C, Sx, Sy, Sa, Sb);
                    node_odd<SM>(Sx, Sy, Sa, Sb, Gx[p], Gy[p], C, q);
                    if constexpr (sizeof(SM) == 2) {
                        V w[8];
                        r0[p] = node_fold_narrow<SM>(d, e[p], q, C, w);
#pragma unroll
                        for (int l = 0; l < 8; ++l) v[l][p] = w[l];
                    } else {
                        r0[p] = node_fold(d, e[p], q);
#pragma unroll
                        for (int l = 0; l < 8; ++l) n[l][p] = q[l];
                    }
                }
            }
            if constexpr (MOM_OUT) {
                auto each = [&](auto fn) {
                    fn(kMomH, H[spp].c);
                    fn(kMomE, e);
                    fn(kMomJx, kx);
                    fn(kMomJy, ky);
                    fn(kMomGx, Gx);
                    fn(kMomGy, Gy);
                };
                const uint32_t off = (uint32_t)y * (uint32_t)mpitch + (uint32_t)xm;
                each([&](int f, const float2(&v)[NP]) { store_group(out0 + f * mplane, off, v); });
                if (odd) each([&](int f, const float2(&v)[NP]) { store_odd(out0 + f * mplane + y * mpitch + 4, true, v); });
            } else {
                const uint32_t off = (uint32_t)y * (uint32_t)pitch + (uint32_t)xg;
                auto each = [&](auto fn) {
#pragma unroll
                    for (int l = 0; l < 8; ++l) {
                        if constexpr (sizeof(SM) == 2) fn(l, v[l]);
                        else fn(l, n[l]);
                    }
                };
                store_group(out0, off, r0);
                each([&](int l, const auto(&q)[NP]) { store_group(outm + plane_of(l) * plane, off, q); });
                if (odd) {
                    store_odd(out0 + y * pitch, false, r0);
                    each([&](int l, const auto(&q)[NP]) { store_odd(outm + plane_of(l) * plane + y * pitch, false, q); });
                }
            }
        }
    };
    for (int k = 0;;) {
        body(std::integral_constant<int, 0>{}, k);
        if (++k > last) break;
        body(std::integral_constant<int, 1>{}, k);
        if (++k > last) break;
        body(std::integral_constant<int, 2>{}, k);
        if (++k > last) break;
    }
}

// 168 registers, twelve warps an SM (13 or 14 spill: 43.6 -> 59.5 and 61.4 us a
// 2048^2 FP32 step with pairs of columns; one pair a thread and 24 warps: 45.8).
template <typename SM, bool MOM_IN, bool MOM_OUT, bool QUAD>
__global__ void __launch_bounds__(32, 12)
k_step4(const void* __restrict__ fin, void* __restrict__ fout, const float* __restrict__ kappa, const Geom G,
        const Consts<float> C)
{
    dependent_launch_entry();
    step_band4<SM, MOM_IN, MOM_OUT, QUAD>(fin, fout, kappa, G, C, blockIdx.x, blockIdx.y, gridDim.y);
}

// Batched form: CTA i takes work item i, a band of a strip (of kWideCols
// columns) of one domain.  QUAD only: the ragged layout lost to the two-column
// march in batches of every size (us a step: 4 domains of 122 x 61 15.3 / 23.1, 64
// of 250 x 125 36 / 62, 16 of 1018 x 509 102 / 155).
template <typename SM, bool MOM_IN, bool MOM_OUT>
__global__ void __launch_bounds__(32, 12)
k_step4_batch(const BatchItem* __restrict__ items, const BatchDomain<float>* __restrict__ doms, int parity)
{
    dependent_launch_entry();
    const BatchItem it = items[blockIdx.x];
    const BatchDomain<float>& D = doms[it.dom];
    const Geom G = D.G;
    Consts<float> C = D.C;
    C.flip = parity;
    step_band4<SM, MOM_IN, MOM_OUT, true>(D.buf[parity], D.buf[parity ^ 1], D.kappa, G, C, it.strip, it.band, it.nbands);
}

}  // namespace tflbm
