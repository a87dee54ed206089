// Paired-column fused step: the same time step as step_band (Section II of
// Zitz et al., arXiv:1810.07642: Eqs. LBE, equilibria, force, pfilm,
// disjoiningP, forcefric, alphafric, derivative, n_laplace), arranged so that
// each thread owns two adjacent lattice columns.
//
// Why: the one-column kernel issues about ten warp instructions per node and
// is limited by instruction issue, not by HBM.  Two columns per thread halve
// the per-node cost of addressing, loop control and barriers, turn every
// population load and store into one aligned 8-byte (FP32) or 4-byte (16-bit
// pair) access, and let the node arithmetic run on Blackwell's paired FP32
// instructions (two lanes of float math per issued instruction).
//
// Storage units.  16-bit storage keeps v_l = (f_l - R_l) * scale for the
// moving populations (R_l the rest equilibrium at href, scale a power of 2).
// The kernel computes on v_l as decoded (one conversion, no arithmetic):
// sums of moving populations need the R_l only through their total 4 (R_axis
// + R_diag), momenta not at all (the R_l are symmetric), and the collision
// forms (f*_l - R_l) * scale directly, with scale and R_l folded into its
// constants.  FP32 storage is the case scale = 1, R_l = 0.
//
// Streaming without misaligned loads.  Thread t loads the nine planes at its
// own aligned column pair (c, c+1).  Populations with c_x = 0 arrive from the
// same columns.  Those with c_x = +1 (l = 1, 2, 8) arrive from the column to
// the left and those with c_x = -1 (l = 4, 5, 6) from the right, so only one
// value per direction crosses a pair boundary.  At tau = 1 the collision
// needs h and j alone, so each thread first sums the three c_x = +1 and the
// three c_x = -1 populations of its own columns; per row four warp shuffles
// then move those two sums and their y-momenta across the pair boundary
// (general tau: six shuffles of the single values, which the relaxation
// needs).  Lane 0 and lane 31 of every warp read the three elements of their
// outer neighbour column themselves (predicated loads that hit L1/L2).
//
// Stencils.  The h and p rows live in 4-row shared rings at their own
// columns; a thread reads its pair as one aligned 8-byte load and the two
// outer neighbours as single values.  (A second, column-shifted copy of each
// row, which would make the shifted pairs aligned loads too, measured slower:
// its extra stores and shared memory cost more than the register moves they
// save.)
//
// Rows, bands, march direction, the reference-height storage and the exact
// mass folding are those of step_band (tflbm_step.cuh).  Needs nx even
// (pairs never straddle the periodic seam); compute type FP32, storage FP32,
// FP16 or BF16.
#pragma once
#include "tflbm_node.cuh"

namespace tflbm {

template <typename V> __device__ __forceinline__ V ldpair(const V* p) { return __ldg(p); }
__device__ __forceinline__ float2 lds2(const float* p) { return *reinterpret_cast<const float2*>(p); }

// the window of an aligned column pair: rows n, c, s of a ring; j is the slot
// of the pair's first column
__device__ __forceinline__ Win<float2> load_win(const float* rn, const float* rc, const float* rs, int j)
{
    Win<float2> w;
    w.n0 = lds2(rn + j); w.nL = make_float2(rn[j - 1], w.n0.x); w.nR = make_float2(w.n0.y, rn[j + 2]);
    w.c0 = lds2(rc + j); w.cL = make_float2(rc[j - 1], w.c0.x); w.cR = make_float2(w.c0.y, rc[j + 2]);
    w.s0 = lds2(rs + j); w.sL = make_float2(rs[j - 1], w.s0.x); w.sR = make_float2(w.s0.y, rs[j + 2]);
    return w;
}

// ---------------------------------------------------------------------------
// One CTA of BX threads covers NC = 2 BX consecutive columns x0-2 .. x0+NC-3
// (thread t: local columns j = 2t, 2t+1) and marches down a band of rows;
// neighbouring CTAs overlap by 4 columns and each stores NC - 4.  The march
// is step_band's: step k forms h of row r(k) into a 4-row shared ring, one
// barrier, then the pressure of row r(k-1) and force, collision and store of
// row r(k-3).  The pulled values of row r(k) come from registers loaded
// one or two rows ahead, plus warp shuffles for the values that cross a pair
// boundary.
template <typename SM, int BX, bool OMEGA1, bool KFIELD>
__device__ __forceinline__ void step_band2(const float* __restrict__ fin0, const SM* __restrict__ finm,
                                           float* __restrict__ fout0, SM* __restrict__ foutm,
                                           const float* __restrict__ kappa, const Geom& G,
                                           const Consts<float>& C, int strip, int band, int nbands)
{
    using IO = PairIO<SM>;
    using V = typename IO::V;
    constexpr bool NARROW = !std::is_same<SM, float>::value;
    constexpr int NC = 2 * BX;  // columns per CTA
    constexpr int W = NC - 4;   // output columns per CTA
    constexpr int OFF = 2;      // ring slot of local column j is OFF + j (keeps pairs 8-byte aligned)
    constexpr int RW = NC + 4;  // ring row width
    // h - href and the film pressure (slot OFF + j: local column j)
    __shared__ __align__(16) float hsm[4][RW];
    __shared__ __align__(16) float psm[4][RW];
    // general tau: the eight pulled moving populations of the last four rows
    __shared__ __align__(16) float2 fsm[OMEGA1 ? 1 : 4][8][OMEGA1 ? 1 : BX];
    // per-thread rings of (j_x, j_y), the pull-sum residual and 1/h of the
    // last four rows (each thread reads back only its own slots)
    __shared__ __align__(16) float4 rsj[4][BX];
    __shared__ __align__(16) float2 rse[4][BX], rsi[4][BX];

    const int t = threadIdx.x, lane = t & 31;
    const int nx = G.nx, ny = G.ny, pitch = G.pitch, plane = (int)G.plane;
    const int x0 = strip * W;
    const int weff = min(W, nx - x0);     // output columns of this CTA (even)
    const bool pcol = 2 * t <= weff + 2;  // p needed at local columns 1 .. weff+2
    const bool ocol = t >= 1 && 2 * t <= weff;
    const int ybeg = (int)(((long long)band * ny) / nbands);
    const int yend = (int)(((long long)(band + 1) * ny) / nbands);
    const int dir = ((band + C.flip) & 1) ? -1 : 1;  // reversed every other step (see make_band)
    const int R = yend - ybeg;
    const int rstart = dir > 0 ? ybeg - 2 : yend + 1;
    const bool disj = KFIELD || C.kappa_u != 0.0f;
    const int c = wrap_index(x0 - 2 + 2 * t, nx);  // own pair (even)
    const int j2 = OFF + 2 * t;                    // ring slot of the pair

    const bool edge = lane == 0 || lane == 31;
    // the outer neighbour column: c - 1 for lane 0, c + 2 for lane 31
    const int ce = lane == 0 ? (c == 0 ? nx - 1 : c - 1) : (c + 2 == nx ? 0 : c + 2);
    // moving planes (index l - 1) a warp-edge lane reads at that column, from
    // rows y, y-1, y+1: lane 0 needs l = 1, 2, 8 (arriving from the left),
    // lane 31 needs l = 5, 4, 6 (from the right)
    const int e0 = (lane == 0 ? 0 : 4) * plane + ce;
    const int e1 = (lane == 0 ? 1 : 3) * plane + ce;
    const int e2 = (lane == 0 ? 7 : 5) * plane + ce;
    const float2* __restrict__ f0p = reinterpret_cast<const float2*>(fin0);
    const V* __restrict__ fmp = reinterpret_cast<const V*>(finm);
    const int half = plane >> 1;  // pairs per plane (pitch is even)
    // PF rows of loads in flight: 16-bit storage keeps two (rows r(k+1) and
    // r(k+2) go out while step k runs), FP32 one (its registers would
    // otherwise cost resident warps)
    constexpr int PF = NARROW ? 2 : 1;
    float2 q0[PF];
    V qm[PF][8];
    SM qe[PF][3];

    // wrapped rows r(k-1) .. r(k+3)
    int wm1 = wrap_index(rstart - dir, ny), w0 = wrap_index(rstart, ny);
    int w1 = wrap_index(rstart + dir, ny), w2 = wrap_index(rstart + 2 * dir, ny);
    int w3 = wrap_index(rstart + 3 * dir, ny);
    // the nine planes (and the edge elements) pulled into row w, into register set b
    auto load_row = [&](auto b_c, int wb, int w, int wa) {
        constexpr int b = decltype(b_c)::value;
        const int ys = dir > 0 ? wb : wa, yn = dir > 0 ? wa : wb;  // rows y-1, y+1
        const int i0 = (w * pitch + c) >> 1, is = (ys * pitch + c) >> 1, in = (yn * pitch + c) >> 1;
        const long long m8 = 8LL * half;  // pairs of the eight moving planes
        int* st = C.status;
        q0[b] = ldpair(f0p + TFLBM_IDX(i0, half, st));
        qm[b][0] = ldpair(fmp + TFLBM_IDX(i0, m8, st));               // l = 1 from row y
        qm[b][1] = ldpair(fmp + TFLBM_IDX(half + is, m8, st));        // l = 2 from row y-1
        qm[b][2] = ldpair(fmp + TFLBM_IDX(2 * half + is, m8, st));    // l = 3
        qm[b][3] = ldpair(fmp + TFLBM_IDX(3 * half + is, m8, st));    // l = 4
        qm[b][4] = ldpair(fmp + TFLBM_IDX(4 * half + i0, m8, st));    // l = 5 from row y
        qm[b][5] = ldpair(fmp + TFLBM_IDX(5 * half + in, m8, st));    // l = 6 from row y+1
        qm[b][6] = ldpair(fmp + TFLBM_IDX(6 * half + in, m8, st));    // l = 7
        qm[b][7] = ldpair(fmp + TFLBM_IDX(7 * half + in, m8, st));    // l = 8
        if (edge) {
            const long long e8 = 8LL * plane;
            qe[b][0] = ldro(finm + TFLBM_IDX(e0 + w * pitch, e8, st));
            qe[b][1] = ldro(finm + TFLBM_IDX(e1 + ys * pitch, e8, st));
            qe[b][2] = ldro(finm + TFLBM_IDX(e2 + yn * pitch, e8, st));
            (void)e8;
        }
        (void)m8;
        (void)st;
    };

    float2 kap_n = pk(C.kappa_u);
    load_row(std::integral_constant<int, 0>{}, wm1, w0, w1);
    if constexpr (PF == 2) load_row(std::integral_constant<int, 1>{}, w0, w1, w2);
    const long long npair = (long long)nx * ny / 2;  // kappa field extent in pairs (nx even)
    (void)npair;
    if (KFIELD && pcol)
        kap_n = reinterpret_cast<const float2*>(kappa)[TFLBM_IDX(((long long)wm1 * nx + c) >> 1, npair, C.status)];

    // ring slots no thread writes: columns -1 and NC (outer halves of the
    // edge columns' stencils)
    if (t < 2) {
        const int j = t == 0 ? OFF - 1 : OFF + NC;
#pragma unroll
        for (int s = 0; s < 4; ++s) hsm[s][j] = psm[s][j] = 0.0f;
    }

    auto body = [&](auto stage_c, int k) {
        constexpr int s = decltype(stage_c)::value;  // ring slot of row r(k)
        constexpr int s1 = (s + 3) & 3;              // r(k-1)
        constexpr int s2 = (s + 2) & 3;              // r(k-2)
        constexpr int s3 = (s + 1) & 3;              // r(k-3)
        const float2 kap = kap_n;                    // kappa of row r(k-1)
        // ---- (A) h, j of row r(k)
        if (k <= R + 3) {
            constexpr int rb = s % PF;  // register set of row r(k)
            const float2 f0 = q0[rb];   // f_0 - href
            float2 v[8];                // moving populations at the own columns, storage units
#pragma unroll
            for (int l = 0; l < 8; ++l) v[l] = IO::dec(qm[rb][l]);
            // the three crossing populations at the outer column (warp-edge lanes)
            float ea = 0.f, eb = 0.f, ed = 0.f;
            if (edge) {
                ea = IO::dec1(qe[rb][0]);  // l = 1 or 5
                eb = IO::dec1(qe[rb][1]);  // l = 2 or 4
                ed = IO::dec1(qe[rb][2]);  // l = 8 or 6
            }
            // the loads of row r(k+PF) go out before this row's arithmetic;
            // at tau = 1 right after the partial sums, which free the
            // registers they land in (FP32 values are used as loaded), so the
            // loads neither wait for nor copy this row (one box, 2048^2 step:
            // FP32 56.0 -> 52.7 us, long-scoreboard stalls 5.3 -> 3.8 per
            // issue; FP16 46.5 -> 45.3 us, BF16 47.1 -> 45.4 us)
            auto issue_next = [&]() {
                if constexpr (PF == 2) {
                    if (k + 2 <= R + 3) load_row(std::integral_constant<int, rb>{}, w1, w2, w3);
                } else {
                    if (k + 1 <= R + 3) load_row(std::integral_constant<int, rb>{}, w0, w1, w2);
                }
            };
            constexpr bool EARLY = !OMEGA1;
            if constexpr (EARLY) issue_next();
            if (KFIELD && pcol)
                kap_n = reinterpret_cast<const float2*>(kappa)[TFLBM_IDX(((long long)w0 * nx + c) >> 1, npair,
                                                                          C.status)];
            // Rs, Ls: sums of the populations arriving from the left (l = 1,
            // 2, 8) and from the right (l = 4, 5, 6) at the two nodes; s26:
            // l = 3, 7; jyr: their y momentum (storage units)
            float2 Rs, Ls, s26, jyr;
            if constexpr (OMEGA1) {
                const float2 Pc = padd(v[0], padd(v[1], v[7])), Py = psub(v[1], v[7]);
                const float2 Qc = padd(v[4], padd(v[3], v[5])), Qy = psub(v[3], v[5]);
                const float2 d26 = psub(v[2], v[6]);
                s26 = padd(v[2], v[6]);
                const float es = ea + (eb + ed), ey = eb - ed;
                if constexpr (!EARLY) issue_next();
                float pl = __shfl_up_sync(0xffffffffu, Pc.y, 1), pyl = __shfl_up_sync(0xffffffffu, Py.y, 1);
                float qr = __shfl_down_sync(0xffffffffu, Qc.x, 1), qyr = __shfl_down_sync(0xffffffffu, Qy.x, 1);
                if (lane == 0) { pl = es; pyl = ey; }
                if (lane == 31) { qr = es; qyr = ey; }
                Rs = make_float2(pl, Pc.x);
                Ls = make_float2(Qc.y, qr);
                jyr = padd(d26, padd(make_float2(pyl, Py.x), make_float2(Qy.y, qyr)));
            } else {
                // the single arriving values, kept for the relaxation
                float u1 = __shfl_up_sync(0xffffffffu, v[0].y, 1);
                float u2 = __shfl_up_sync(0xffffffffu, v[1].y, 1);
                float u8 = __shfl_up_sync(0xffffffffu, v[7].y, 1);
                float d5 = __shfl_down_sync(0xffffffffu, v[4].x, 1);
                float d4 = __shfl_down_sync(0xffffffffu, v[3].x, 1);
                float d6 = __shfl_down_sync(0xffffffffu, v[5].x, 1);
                if (lane == 0) { u1 = ea; u2 = eb; u8 = ed; }
                if (lane == 31) { d5 = ea; d4 = eb; d6 = ed; }
                float2 n[8];
                n[0] = make_float2(u1, v[0].x);
                n[1] = make_float2(u2, v[1].x);
                n[2] = v[2];
                n[3] = make_float2(v[3].y, d4);
                n[4] = make_float2(v[4].y, d5);
                n[5] = make_float2(v[5].y, d6);
                n[6] = v[6];
                n[7] = make_float2(u8, v[7].x);
                Rs = padd(n[0], padd(n[1], n[7]));
                Ls = padd(n[4], padd(n[3], n[5]));
                jyr = padd(psub(n[2], n[6]), padd(psub(n[1], n[7]), psub(n[3], n[5])));
                s26 = padd(n[2], n[6]);
#pragma unroll
                for (int l = 0; l < 8; ++l) fsm[s][l][t] = n[l];
            }
            float2 dh, er, jx, jy;
            node_moments<SM>(f0, Rs, Ls, s26, jyr, C, dh, er, jx, jy);
            TFLBM_CHECK(j2 >= OFF && j2 + 1 < RW, C.status);
            *reinterpret_cast<float2*>(&hsm[s][j2]) = dh;
            rsj[s][t] = make_float4(jx.x, jx.y, jy.x, jy.y);
            rse[s][t] = er;
        }
        __syncthreads();
        // ---- (B1) film pressure of row r(k-1) (needs h rows r(k-2) .. r(k))
        if (pcol && k >= 2 && k <= R + 3) {
            // the window reads slots j2 - 1 .. j2 + 2 of rings of RW
            TFLBM_CHECK(j2 >= 1 && j2 + 2 < RW, C.status);
            float2 ih;
            const Win<float2> Hw = load_win(hsm[s], hsm[s1], hsm[s2], j2);
            const float2 p = node_pressure(Hw, kap, disj, C, ih);
            rsi[s1][t] = ih;
            *reinterpret_cast<float2*>(&psm[s1][j2]) = p;
        }
        // ---- (B2) force, collision and store of row r(k-3)
        if (ocol && k >= 5) {
            const int o = rstart + (k - 3) * dir;  // inside [ybeg, yend), no wrap
            TFLBM_CHECK(j2 >= 1 && j2 + 2 < RW && o >= 0 && o < ny, C.status);
            // rows o+1 and o-1 of the p ring
            const int sn = dir > 0 ? s2 : s, ss = dir > 0 ? s : s2;
            const Win<float2> Pw = load_win(psm[sn], psm[s3], psm[ss], j2);
            const float2 dh = lds2(&hsm[s3][j2]);
            const float4 jj = rsj[s3][t];
            const float2* fp = nullptr;
            if constexpr (!OMEGA1) fp = &fsm[s3][0][t];
            // the pair (i, i+1) of plane 0 and of the eight moving planes
            const int i = o * pitch + c;
            TFLBM_CHECK(i >= 0 && (i & 1) == 0 && i + 1 < plane, C.status);
            const int ip = TFLBM_IDX(i >> 1, half, C.status);
            node_collide<SM, OMEGA1>(Pw, dh, rsi[s3][t], make_float2(jj.x, jj.y), make_float2(jj.z, jj.w), rse[s3][t],
                                     fp, BX, C, [&](float2 o0, const V(&q)[8]) {
                                         reinterpret_cast<float2*>(fout0)[ip] = o0;
                                         V* om = reinterpret_cast<V*>(foutm) + ip;
#pragma unroll
                                         for (int l = 0; l < 8; ++l) om[l * half] = q[l];
                                     });
        }
        wm1 = w0;
        w0 = w1;
        w1 = w2;
        w2 = w3;
        w3 += dir;
        w3 = w3 == ny ? 0 : (w3 < 0 ? ny - 1 : w3);
    };

    const int last = R + 4;
    for (int k = 0;;) {
        body(std::integral_constant<int, 0>{}, k);
        if (++k > last) break;
        body(std::integral_constant<int, 1>{}, k);
        if (++k > last) break;
        body(std::integral_constant<int, 2>{}, k);
        if (++k > last) break;
        body(std::integral_constant<int, 3>{}, k);
        if (++k > last) break;
    }
}

// Register budget: 80 per thread (24 resident warps per SM), at which the
// kernel does not spill (measured faster than 128 registers and 16 warps).
template <typename SM, int BX, bool OMEGA1, bool KFIELD>
__global__ void __launch_bounds__(BX, 768 / BX)
k_step2(const float* __restrict__ fin0, const SM* __restrict__ finm, float* __restrict__ fout0,
        SM* __restrict__ foutm, const float* __restrict__ kappa, const Geom G, const Consts<float> C)
{
    dependent_launch_entry();
    step_band2<SM, BX, OMEGA1, KFIELD>(fin0, finm, fout0, foutm, kappa, G, C, blockIdx.x, blockIdx.y, gridDim.y);
}

// ---------------------------------------------------------------------------
// Batched form: the work items of k_step_batch (a band of a strip of one
// domain; block_x columns per strip in both kernels), each run as
// step_band2 with its domain's geometry and constants.  Every domain reads
// its buffer `parity` and writes the other one; queue as in k_step_batch (a
// persistent grid taking items from a counter, reset by the last CTA; no CTA
// waits on another).  Needs every domain's nx even and the FP32 compute type.
template <typename SM, int BX, bool OMEGA1, bool KFIELD>
__device__ __forceinline__ void batch_item2(const BatchItem it, const BatchDomain<float>* __restrict__ doms,
                                            int parity)
{
    const BatchDomain<float>& D = doms[it.dom];
    const Geom G = D.G;
    Consts<float> C = D.C;
    C.flip = parity;
    const void* fin = D.buf[parity];
    void* fout = D.buf[parity ^ 1];
    const float* f0 = (const float*)fin;
    const SM* fm = (const SM*)((const char*)fin + G.plane * sizeof(float));
    float* g0 = (float*)fout;
    SM* gm = (SM*)((char*)fout + G.plane * sizeof(float));
    step_band2<SM, BX, OMEGA1, KFIELD>(f0, fm, g0, gm, D.kappa, G, C, it.strip, it.band, it.nbands);
}

template <typename SM, int BX, bool OMEGA1, bool KFIELD>
__global__ void __launch_bounds__(BX, 768 / BX)
k_step2_batch(const BatchItem* __restrict__ items, int nitems, const BatchDomain<float>* __restrict__ doms,
              int parity, int* queue)
{
    dependent_launch_entry();
    if (!queue) {
        batch_item2<SM, BX, OMEGA1, KFIELD>(items[blockIdx.x], doms, parity);
        return;
    }
    __shared__ int next;
    for (;;) {
        __syncthreads();  // the previous item is done with the shared rings and with `next`
        if (threadIdx.x == 0) next = atomicAdd(queue, 1);
        __syncthreads();
        const int i = next;
        if (i >= nitems) break;
        batch_item2<SM, BX, OMEGA1, KFIELD>(items[i], doms, parity);
    }
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(queue + 1, 1) == (int)gridDim.x - 1) {  // every CTA has taken its last item
            queue[0] = 0;
            queue[1] = 0;
        }
    }
}

template <typename SM, int BX, bool OM1, bool KF>
cudaError_t batch2_one(const BatchLaunch& L, cudaStream_t st)
{
    const BatchDomain<float>* d = (const BatchDomain<float>*)L.doms;
    if (L.query_occupancy) {
        int n = 0;
        const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_step2_batch<SM, BX, OM1, KF>, BX, 0);
        *L.query_occupancy = e == cudaSuccess ? n : 0;
        return e;
    }
    return launch_dependent(k_step2_batch<SM, BX, OM1, KF>, dim3(L.grid), BX, 0, st, L.items, L.nitems, d, L.parity,
                            L.queue);
}

// The batched paired step for one storage type (L.block_x columns per CTA).
template <typename SM>
cudaError_t pair_step_batch(const BatchLaunch& L, cudaStream_t st)
{
    auto pick = [&](auto bx_c) {
        constexpr int BX = decltype(bx_c)::value;
        if (L.kfield) return L.omega1 ? batch2_one<SM, BX, true, true>(L, st) : batch2_one<SM, BX, false, true>(L, st);
        return L.omega1 ? batch2_one<SM, BX, true, false>(L, st) : batch2_one<SM, BX, false, false>(L, st);
    };
    switch (L.block_x) {
        case 64: return pick(std::integral_constant<int, 32>{});
        case 128: return pick(std::integral_constant<int, 64>{});
        case 256: return pick(std::integral_constant<int, 128>{});
        default: return cudaErrorInvalidValue;
    }
}

// ---------------------------------------------------------------------------
// Launch of the paired kernel: block_x is the CTA width in columns (64, 128
// or 256), i.e. block_x / 2 threads.

template <typename SM, int BX>
cudaError_t launch_pair_bx(const float* fin0, const SM* finm, float* fout0, SM* foutm, const float* kappa,
                           const Geom& G, const Consts<float>& C, int bands, cudaStream_t st)
{
    constexpr int W = 2 * BX - 4;
    const dim3 grid((G.nx + W - 1) / W, bands);
    const bool om1 = C.omega == 1.0f;
    if (kappa) {
        if (om1) return launch_dependent(k_step2<SM, BX, true, true>, grid, BX, 0, st, fin0, finm, fout0, foutm, kappa, G, C);
        return launch_dependent(k_step2<SM, BX, false, true>, grid, BX, 0, st, fin0, finm, fout0, foutm, kappa, G, C);
    }
    if (om1) return launch_dependent(k_step2<SM, BX, true, false>, grid, BX, 0, st, fin0, finm, fout0, foutm, kappa, G, C);
    return launch_dependent(k_step2<SM, BX, false, false>, grid, BX, 0, st, fin0, finm, fout0, foutm, kappa, G, C);
}

template <typename SM, int BX, bool OM1, bool KF>
int bps_pair_one()
{
    int n = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_step2<SM, BX, OM1, KF>, BX, 0);
    return e == cudaSuccess ? n : 0;
}

// The paired step for one storage type.
template <typename SM>
cudaError_t pair_step(int block_x, const void* fin, void* fout, const void* kappa, const Geom& G,
                      const Consts<float>& C, int bands, cudaStream_t st)
{
    const float* f0 = (const float*)fin;
    const SM* fm = (const SM*)((const char*)fin + G.plane * sizeof(float));
    float* g0 = (float*)fout;
    SM* gm = (SM*)((char*)fout + G.plane * sizeof(float));
    const float* k = (const float*)kappa;
    switch (block_x) {
        case 64: return launch_pair_bx<SM, 32>(f0, fm, g0, gm, k, G, C, bands, st);
        case 128: return launch_pair_bx<SM, 64>(f0, fm, g0, gm, k, G, C, bands, st);
        case 256: return launch_pair_bx<SM, 128>(f0, fm, g0, gm, k, G, C, bands, st);
        default: return cudaErrorInvalidValue;
    }
}

// Resident CTAs per SM of the paired step for a CTA width (0 if unknown).
template <typename SM>
int pair_blocks_per_sm(int block_x, bool omega1, bool kfield)
{
    auto pick = [&](auto bx_c) {
        constexpr int BX = decltype(bx_c)::value;
        if (kfield) return omega1 ? bps_pair_one<SM, BX, true, true>() : bps_pair_one<SM, BX, false, true>();
        return omega1 ? bps_pair_one<SM, BX, true, false>() : bps_pair_one<SM, BX, false, false>();
    };
    switch (block_x) {
        case 64: return pick(std::integral_constant<int, 32>{});
        case 128: return pick(std::integral_constant<int, 64>{});
        case 256: return pick(std::integral_constant<int, 128>{});
        default: return 0;
    }
}

}  // namespace tflbm
