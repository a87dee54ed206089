// Auxiliary kernels of the thin-film D2Q9 library: kappa field, initial
// populations, moments, film pressure and force (diagnostic), compensated
// mass, state scan and state import/export.
//
// The stored buffer holds post-collision (pre-streaming) populations B_l, so
// the post-streaming populations of the current time are f_l(x) = B_l(x - c_l).
// Plane 0 stores B_0 - href in the compute type; the 8 moving planes follow in
// the storage type (the compute type, or a 16-bit encoding, see Consts in
// tflbm_internal.h).  All kernels here go through the Pops accessor below.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <math.h>

#include <type_traits>

#include "tflbm_internal.h"

namespace tflbm {
namespace {

// Velocities of Eq. (speeds).  Functions of an unrolled index rather than
// __constant__ arrays: they fold to literals, so a pull needs three wrapped
// rows and three wrapped columns instead of eighteen runtime ones.
__host__ __device__ constexpr int cx_of(int l) { return l == 1 || l == 2 || l == 8 ? 1 : (l >= 4 && l <= 6 ? -1 : 0); }
__host__ __device__ constexpr int cy_of(int l) { return l >= 2 && l <= 4 ? 1 : (l >= 6 ? -1 : 0); }

// i in [-1, n] on a ring of n (a compare each way; the integer modulo this
// replaces cost more than the loads it indexed: plot-file read-out of 2048^2,
// moments + pressure and force, 250 -> 93 us together with the fused k_pf).
__device__ __forceinline__ int wrapi(int i, int n) { return i < 0 ? n - 1 : (i >= n ? 0 : i); }

// Wrapped columns x-1, x, x+1 and row offsets of y-1, y, y+1 (rows of `pitch`
// elements).
struct Around {
    int x[3], r[3];  // 32-bit: 9 planes stay below 2^31 elements
    __device__ __forceinline__ Around(int x_, int y_, int nx, int ny, int pitch)
    {
        x[0] = wrapi(x_ - 1, nx);
        x[1] = x_;
        x[2] = wrapi(x_ + 1, nx);
        r[0] = wrapi(y_ - 1, ny) * pitch;
        r[1] = y_ * pitch;
        r[2] = wrapi(y_ + 1, ny) * pitch;
    }
    // element of the node (dx, dy) away, dx, dy in {-1, 0, 1}
    __device__ __forceinline__ int at(int dx, int dy) const { return r[dy + 1] + x[dx + 1]; }
};

__device__ __forceinline__ float cvt(float q) { return q; }
__device__ __forceinline__ double cvt(double q) { return q; }
__device__ __forceinline__ float cvt(__half q) { return __half2float(q); }
__device__ __forceinline__ float cvt(__nv_bfloat16 q) { return __bfloat162float(q); }
template <typename SM> __device__ __forceinline__ SM enc(float v);
template <> __device__ __forceinline__ __half enc<__half>(float v) { return __float2half_rn(v); }
template <> __device__ __forceinline__ __nv_bfloat16 enc<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// Read / write access to one population buffer.
template <typename T, typename SM>
struct Pops {
    T* f0;       // plane 0: f_0 - href
    SM* fm;      // moving planes 1..8
    int plane, pitch;
    T href, mscale, minv, r_axis, r_diag;

    __device__ __forceinline__ int at(int y, int x) const { return y * pitch + x; }
    // the stored value of plane l at element i, decoded (plane 0: f_0 - href)
    __device__ __forceinline__ T raw(int l, int i) const
    {
        if (l == 0) return f0[i];
        const SM q = fm[(l - 1) * plane + i];
        if constexpr (std::is_same<SM, T>::value) return q;
        else return fmaf(cvt(q), minv, (l & 1) ? r_axis : r_diag);
    }
    __device__ __forceinline__ T full(int l, int i) const { return l == 0 ? raw(0, i) + href : raw(l, i); }
    // store the population value v (plane 0: v is f_0 - href)
    __device__ __forceinline__ void put(int l, int i, T v) const
    {
        if (l == 0) f0[i] = v;
        else if constexpr (std::is_same<SM, T>::value) fm[(l - 1) * plane + i] = v;
        else fm[(l - 1) * plane + i] = enc<SM>((v - ((l & 1) ? r_axis : r_diag)) * mscale);
    }
};

template <typename T, typename SM>
Pops<T, SM> make_pops(const void* buf, const Geom& G, const StoreDesc& D)
{
    Pops<T, SM> P;
    P.f0 = (T*)buf;
    P.fm = (SM*)((char*)buf + G.plane * sizeof(T));
    P.plane = (int)G.plane;
    P.pitch = G.pitch;
    P.href = T(D.href);
    P.mscale = T(D.mscale);
    P.minv = T(D.minv);
    P.r_axis = T(D.r_axis);
    P.r_diag = T(D.r_diag);
    return P;
}

// Post-streaming populations at (x, y).
template <typename T, typename SM>
__device__ __forceinline__ void pull_at(const Pops<T, SM>& P, const Geom& G, int x, int y, T (&v)[9])
{
    const Around N(x, y, G.nx, G.ny, P.pitch);
#pragma unroll
    for (int l = 0; l < 9; ++l) v[l] = P.full(l, N.at(-cx_of(l), -cy_of(l)));
}

template <typename T>
__device__ __forceinline__ void moments9(const T (&v)[9], T& h, T& jx, T& jy)
{
    h = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7])) + v[8];
    jx = ((v[1] + v[2]) + v[8]) - ((v[4] + v[5]) + v[6]);
    jy = ((v[2] + v[3]) + v[4]) - ((v[6] + v[7]) + v[8]);
}

// kappa(x) = (1 - cos theta)(n-1)(m-1)/((n-m) h_*), Eq. (disjoiningP), in double.
template <typename T>
__global__ void k_kappa(T* kappa, const T* theta, long long n, int ne, int me, double hstar)
{
    const double c = (double)(ne - 1) * (double)(me - 1) / ((double)(ne - me) * hstar);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        kappa[i] = T((1.0 - cos((double)theta[i])) * c);
}

// B_l(x) = f_eq_l(h0(x + c_l), u = 0), so that the pull gives f = f_eq(h0, 0).
template <typename T, typename SM>
__global__ void k_init(Pops<T, SM> P, const T* __restrict__ h0, Geom G, T g)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= G.nx) return;
    const Around N(x, y, G.nx, G.ny, G.nx);
#pragma unroll
    for (int l = 0; l < 9; ++l) {
        const T h = h0[N.at(cx_of(l), cy_of(l))];
        const T gh2 = g * h * h;
        T v;
        if (l == 0) v = (h - P.href) - T(5.0 / 6.0) * gh2;
        else if (l & 1) v = gh2 * T(1.0 / 6.0);
        else v = gh2 * T(1.0 / 24.0);
        P.put(l, P.at(y, x), v);
    }
}

template <typename T, typename SM>
__global__ void k_moments(Pops<T, SM> P, T* h, T* ux, T* uy, Geom G)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= G.nx) return;
    T v[9], hh, jx, jy;
    pull_at(P, G, x, y, v);
    moments9(v, hh, jx, jy);
    const long long i = (long long)y * G.nx + x;
    if (h) h[i] = hh;
    if (ux) ux[i] = jx / hh;
    if (uy) uy[i] = jy / hh;
}

template <typename T>
__device__ __forceinline__ T ipow_(T r, int n)
{
    T o = T(1);
    for (int i = 0; i < n; ++i) o *= r;
    return o;
}

template <typename T>
__global__ void k_pf_p(const T* __restrict__ hbuf, const T* __restrict__ kappa, T* pbuf, Geom G,
                       Consts<T> C)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= G.nx) return;
    const int xm = wrapi(x - 1, G.nx), xp = wrapi(x + 1, G.nx);
    const int ym = wrapi(y - 1, G.ny), yp = wrapi(y + 1, G.ny);
    auto H = [&](int yy, int xx) { return hbuf[(long long)yy * G.nx + xx]; };
    const T h = H(y, x);
    const T axis = H(y, xm) + H(y, xp) + H(ym, x) + H(yp, x);
    const T diag = H(ym, xm) + H(ym, xp) + H(yp, xm) + H(yp, xp);
    T lap = (T(4) * axis + diag - T(20) * h) / T(6);
    const T kap = kappa ? kappa[(long long)y * G.nx + x] : C.kappa_u;
    const T r = C.hstar / h;
    lap += C.pi_sgn * kap * (ipow_(r, C.n_exp) - ipow_(r, C.m_exp));
    pbuf[(long long)y * G.nx + x] = -C.gamma * lap;
}

// i on a ring of n, for the halo of a tile (any i; the modulo runs only
// outside the lattice)
__device__ __forceinline__ int ringi(int i, int n)
{
    if ((unsigned)i < (unsigned)n) return i;
    i %= n;
    return i < 0 ? i + n : i;
}

// Film pressure and force of the current state in one pass.  Bound by HBM (36
// B of populations in, 12 B out a node in FP32) plus the halo's second reads
// from L1/L2; before, three kernels read the populations twice and moved h
// and p through memory.  A CTA owns a tile of kPfX x kPfY nodes: h - href of
// the tile and a halo of 2, the pressure of the tile and a halo of 1, then the
// force; each thread keeps the momenta of its own nodes.  64 x 16: rows
// long enough for coalesced pulls, 1.33 pulls a node.  2048^2 FP32 read-out
// (k_moments and this): 250 -> 93 us.  64 x 4 for FP64 state on lattices of fewer
// 64 x 16 tiles than half the SMs, where a CTA's FP64 arithmetic is a chain on one
// SM (128^2, with the launch: 28 us as three kernels, 38 in 16 rows, 25 in 4).
constexpr int kPfX = 64, kPfThreads = 256;
template <typename T, typename SM, int kPfY>
__global__ void __launch_bounds__(kPfThreads) k_pf(Pops<T, SM> P, const T* __restrict__ kappa, T* p, T* fx, T* fy,
                                                   Geom G, Consts<T> C)
{
    constexpr int kPfOwn = kPfX * kPfY / kPfThreads;
    __shared__ T hs[kPfY + 4][kPfX + 4];
    __shared__ T ps[kPfY + 2][kPfX + 2];
    const int x0 = blockIdx.x * kPfX, y0 = blockIdx.y * kPfY;
    const int w = min(kPfX, G.nx - x0), hgt = min(kPfY, G.ny - y0);
    const int tx = threadIdx.x % kPfX, ty = threadIdx.x / kPfX;
    // h - href of the node at tile position (c, r), and its momentum
    auto pull = [&](int c, int r, T& jx, T& jy) {
        const Around N(ringi(x0 + c, G.nx), ringi(y0 + r, G.ny), G.nx, G.ny, P.pitch);
        T v[9];
#pragma unroll
        for (int l = 0; l < 9; ++l) v[l] = P.raw(l, N.at(-cx_of(l), -cy_of(l)));
        T dh;
        moments9(v, dh, jx, jy);
        return dh;
    };
    auto pressure = [&](int c, int r) {
        const T(&H)[kPfY + 4][kPfX + 4] = hs;
        const int i = r + 2, j = c + 2;
        const T axis = (H[i][j - 1] + H[i][j + 1]) + (H[i - 1][j] + H[i + 1][j]);
        const T diag = (H[i - 1][j - 1] + H[i - 1][j + 1]) + (H[i + 1][j - 1] + H[i + 1][j + 1]);
        T lap = (T(4) * axis + diag - T(20) * H[i][j]) * T(1.0 / 6.0);
        const T kap = kappa ? kappa[ringi(y0 + r, G.ny) * G.nx + ringi(x0 + c, G.nx)] : C.kappa_u;
        const T q = C.hstar / (H[i][j] + P.href);
        const T fd = C.n_exp == 3 && C.m_exp == 2 ? q * q * (q - T(1)) : ipow_(q, C.n_exp) - ipow_(q, C.m_exp);
        lap += C.pi_sgn * kap * fd;
        return -C.gamma * lap;
    };
    T jx[kPfOwn], jy[kPfOwn];
    bool own[kPfOwn];
#pragma unroll
    for (int k = 0; k < kPfOwn; ++k) {
        const int r = ty + k * (kPfThreads / kPfX);
        own[k] = tx < w && r < hgt;
        jx[k] = jy[k] = T(0);
        if (own[k]) hs[r + 2][tx + 2] = pull(tx, r, jx[k], jy[k]);
    }
    // halo of 2: two rows below and above, two columns left and right
    constexpr int HR = 4 * (kPfX + 4);
    for (int i = threadIdx.x; i < HR + 4 * kPfY; i += kPfThreads) {
        int c, r;
        if (i < HR) {
            const int k = i / (kPfX + 4);
            c = i % (kPfX + 4) - 2;
            r = k < 2 ? k - 2 : hgt + k - 2;
        } else {
            const int k = (i - HR) % 4;
            r = (i - HR) / 4;
            c = k < 2 ? k - 2 : w + k - 2;
        }
        T a, b;
        if (c < w + 2 && r < hgt + 2) hs[r + 2][c + 2] = pull(c, r, a, b);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kPfOwn; ++k) {
        const int r = ty + k * (kPfThreads / kPfX);
        if (own[k]) ps[r + 1][tx + 1] = pressure(tx, r);
    }
    constexpr int PR = 2 * (kPfX + 2);
    for (int i = threadIdx.x; i < PR + 2 * kPfY; i += kPfThreads) {
        int c, r;
        if (i < PR) {
            c = i % (kPfX + 2) - 1;
            r = i / (kPfX + 2) == 0 ? -1 : hgt;
        } else {
            r = (i - PR) / 2;
            c = (i - PR) % 2 == 0 ? -1 : w;
        }
        if (c < w + 1 && r < hgt + 1) ps[r + 1][c + 1] = pressure(c, r);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kPfOwn; ++k) {
        const int r = ty + k * (kPfThreads / kPfX);
        if (!own[k]) continue;
        auto Pp = [&](int dy, int dx) { return ps[r + 1 + dy][tx + 1 + dx]; };
        const T third = T(1.0 / 3.0), twelfth = T(1.0 / 12.0);
        const T gpx = (Pp(0, 1) - Pp(0, -1)) * third + (Pp(1, 1) - Pp(1, -1) + Pp(-1, 1) - Pp(-1, -1)) * twelfth;
        const T gpy = (Pp(1, 0) - Pp(-1, 0)) * third + (Pp(1, 1) - Pp(-1, 1) + Pp(1, -1) - Pp(-1, -1)) * twelfth;
        const T hh = hs[r + 2][tx + 2] + P.href;
        const T fr = C.nu6 / (T(2) * hh * hh + T(6) * C.delta * hh + T(3) * C.delta * C.delta);
        const long long i = (long long)(y0 + r) * G.nx + x0 + tx;
        if (p) p[i] = Pp(0, 0);
        T Fx = -hh * gpx - fr * jx[k] + hh * C.gx;
        T Fy = -hh * gpy - fr * jy[k] + hh * C.gy;
        if (C.forcing) {
            // second-order forcing: friction at u = (j + F/2)/h, i.e.
            // h u (1 + fr/2) = j + F'/2 with F' the force without friction
            const T fpx = hh * (C.gx - gpx), fpy = hh * (C.gy - gpy);
            const T q = T(1) / (T(1) + T(0.5) * fr);
            Fx = fpx - fr * (jx[k] + T(0.5) * fpx) * q;
            Fy = fpy - fr * (jy[k] + T(0.5) * fpy) * q;
        }
        if (fx) fx[i] = Fx;
        if (fy) fy[i] = Fy;
    }
}

// Neumaier pair (s, c): value s + c.
struct Comp {
    double s, c;
};

__device__ __forceinline__ void comp_add(Comp& a, double v)
{
    const double t = a.s + v;
    if (fabs(a.s) >= fabs(v)) a.c += (a.s - t) + v;
    else a.c += (v - t) + a.s;
    a.s = t;
}

__device__ __forceinline__ void comp_merge(Comp& a, const Comp& b)
{
    comp_add(a, b.s);
    a.c += b.c;
}

__device__ __forceinline__ Comp warp_reduce(Comp a)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        Comp b;
        b.s = __shfl_down_sync(0xffffffffu, a.s, off);
        b.c = __shfl_down_sync(0xffffffffu, a.c, off);
        comp_merge(a, b);
    }
    return a;
}

constexpr int kMassThreads = 256;

__device__ __forceinline__ void block_store(Comp a, double* partials)
{
    a = warp_reduce(a);
    __shared__ Comp sm[kMassThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) sm[wid] = a;
    __syncthreads();
    if (wid == 0) {
        Comp b = lane < kMassThreads / 32 ? sm[lane] : Comp{0.0, 0.0};
        b = warp_reduce(b);
        if (lane == 0) {
            partials[2 * blockIdx.x] = b.s;
            partials[2 * blockIdx.x + 1] = b.c;
        }
    }
}

// Sum of every stored population, decoded (the total liquid volume minus
// nx*ny*href: streaming only permutes populations on the periodic lattice).
// With an FP32 compute type each thread keeps an error-free FP32 pair
// (sum, compensation; Knuth's TwoSum per element), which resolves the sum of
// its ~100 values to about 2^-48 and runs at FP32 rate; the pair goes to the
// double-precision block reduction once.  FP64 state sums in double.
template <typename T, typename SM>
__global__ void __launch_bounds__(kMassThreads) k_mass_partial(Pops<T, SM> P, Geom G, double* partials)
{
    Comp a{0.0, 0.0};
    float fs = 0.0f, fc = 0.0f;
    const long long nrows = 9LL * G.ny;
    for (long long row = blockIdx.x; row < nrows; row += gridDim.x) {
        const int l = (int)(row / G.ny), y = (int)(row % G.ny);
        for (int x = threadIdx.x; x < G.nx; x += blockDim.x) {
            const T v = P.raw(l, P.at(y, x));
            if constexpr (std::is_same<T, float>::value) {
                const float t = __fadd_rn(fs, v);
                const float bp = __fsub_rn(t, fs);
                fc = __fadd_rn(fc, __fadd_rn(__fsub_rn(fs, __fsub_rn(t, bp)), __fsub_rn(v, bp)));
                fs = t;
            } else {
                comp_add(a, (double)v);
            }
        }
    }
    if constexpr (std::is_same<T, float>::value) {
        comp_add(a, (double)fs);
        a.c += (double)fc;
    }
    block_store(a, partials);
}

// Thread 0 of the block receives the block's compensated sum / maximum.
__device__ __forceinline__ Comp block_sum(Comp a)
{
    __shared__ Comp sm[kMassThreads / 32];
    a = warp_reduce(a);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();  // sm may still be read from a previous call
    if (lane == 0) sm[wid] = a;
    __syncthreads();
    Comp b{0.0, 0.0};
    if (wid == 0) {
        b = lane < kMassThreads / 32 ? sm[lane] : Comp{0.0, 0.0};
        b = warp_reduce(b);
    }
    return b;
}

__device__ __forceinline__ double block_max(double v)
{
    __shared__ double sm[kMassThreads / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sm[wid] = v;
    __syncthreads();
    double b = -INFINITY;
    if (wid == 0) {
        b = lane < kMassThreads / 32 ? sm[lane] : -INFINITY;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) b = fmax(b, __shfl_xor_sync(0xffffffffu, b, o));
    }
    return b;
}

template <typename T, typename SM>
__device__ __forceinline__ Pops<T, SM> pops_of(const BatchDomain<T>& D, int parity)
{
    Pops<T, SM> P;
    P.f0 = (T*)D.buf[parity];
    P.fm = (SM*)((char*)D.buf[parity] + D.G.plane * sizeof(T));
    P.plane = (int)D.G.plane;
    P.pitch = D.G.pitch;
    P.href = D.C.href;
    P.mscale = D.C.mscale;
    P.minv = D.C.minv;
    P.r_axis = D.C.r_axis;
    P.r_diag = D.C.r_diag;
    return P;
}

// One entry of a domain's trigonometric table: cos and sin of 2 pi i / n, with
// an FP32 compute type as the sum of three floats, which holds all bits of the
// double.  Entries 0 .. nx-1 are the columns, nx .. nx+ny-1 the rows.  A
// Fourier phase 2 pi m x / n is entry m x mod n, so the table does not depend
// on the mode.
template <typename T> struct Trig;
template <> struct __align__(16) Trig<float> {
    float2 hi, lo, lo2, pad;  // (cos, sin)
    __device__ __forceinline__ void set(double c, double s)
    {
        hi = make_float2((float)c, (float)s);
        const double cr = c - (double)hi.x, sr = s - (double)hi.y;
        lo = make_float2((float)cr, (float)sr);
        lo2 = make_float2((float)(cr - (double)lo.x), (float)(sr - (double)lo.y));
        pad = make_float2(0.0f, 0.0f);
    }
    // the factors (-sin, cos)
    __device__ __forceinline__ Trig turned() const
    {
        return {make_float2(-hi.y, hi.x), make_float2(-lo.y, lo.x), make_float2(-lo2.y, lo2.x), pad};
    }
};
template <> struct __align__(16) Trig<double> {
    double2 hi;
    __device__ __forceinline__ void set(double c, double s) { hi = make_double2(c, s); }
    __device__ __forceinline__ Trig turned() const { return {make_double2(-hi.y, hi.x)}; }
};
static_assert(sizeof(Trig<float>) == diag_trig_bytes(false) && sizeof(Trig<double>) == diag_trig_bytes(true),
              "table entry size");

// Running sums of the diagnostics, two at a time.  The reference is sums in
// compensated doubles, whose error is the rounding of the result; but GB300
// retires 2 FP64 operations a clock and SM, and such sums, with a double
// sincospi per node, took 2130 us for 32 domains.  With an FP32 compute type a
// sum is therefore three floats: Knuth's TwoSum of the sum and each addend, of
// its errors and theirs, and a plain sum of the errors of that (as good as a sum
// in three times the precision, rounded once: an error of about n 2^-72 of the
// sum of |addends|, n addends); products are split by fma.  Both sums share
// Blackwell's paired FP32 instructions.  A sum of two floats, without the third,
// loses with its length: 2^-48 of the sum for 16 addends, 2^-44 for 128, 2^-38
// for 8192.  Addends are scaled by kSumScale, so that no sum of a lattice
// overflows where its addends do not.  FP64 state sums in compensated doubles.
constexpr double kSumScale = 1.0 / 4294967296.0;  // 2^-32; fewer than 2^31 nodes
// a - b in one instruction (the paired add takes no negated operand)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
// s += v; returns the rounding error
__device__ __forceinline__ float2 two_sum2(float2& s, float2 v)
{
    const float2 t = __fadd2_rn(s, v), b = sub2(t, s);
    const float2 e = __fadd2_rn(sub2(s, sub2(t, b)), sub2(v, b));
    s = t;
    return e;
}
template <typename T> struct Acc2;
template <> struct Acc2<float> {
    using V = float2;
    static constexpr double kScale = kSumScale;
    V s = {0.0f, 0.0f}, c = {0.0f, 0.0f}, d = {0.0f, 0.0f};
    __device__ __forceinline__ void add(V v) { d = __fadd2_rn(d, two_sum2(c, two_sum2(s, v))); }
    // += v * w
    __device__ __forceinline__ void add_product(V v, const Trig<float>& w)
    {
        // the rounding error of a product, v hi - q, is exact in one fma
        const V q = __fmul2_rn(v, w.hi), r = __fmul2_rn(v, w.lo);
        const V e = two_sum2(c, two_sum2(s, q)), f = two_sum2(c, __ffma2_rn(v, w.hi, V{-q.x, -q.y}));
        const V g = two_sum2(c, r), l = __ffma2_rn(v, w.lo2, __ffma2_rn(v, w.lo, V{-r.x, -r.y}));
        d = __fadd2_rn(d, __fadd2_rn(__fadd2_rn(e, f), __fadd2_rn(g, l)));
    }
    // += the first or second sum of a * w
    __device__ __forceinline__ void add_first(const Acc2& a, const Trig<float>& w) { add_sum(a.s.x, a.c.x, a.d.x, w); }
    __device__ __forceinline__ void add_second(const Acc2& a, const Trig<float>& w) { add_sum(a.s.y, a.c.y, a.d.y, w); }
    __device__ __forceinline__ void merge(const Acc2& a)
    {
        const V e = two_sum2(c, two_sum2(s, a.s));
        d = __fadd2_rn(d, __fadd2_rn(__fadd2_rn(e, two_sum2(c, a.c)), a.d));
    }
    // fn of the values of a and b, part by part
    template <typename Fn>
    static __device__ __forceinline__ Acc2 of(const Acc2& a, const Acc2& b, Fn fn)
    {
        Acc2 r;
        r.s = fn(a.s, b.s);
        r.c = fn(a.c, b.c);
        r.d = fn(a.d, b.d);
        return r;
    }
    __device__ __forceinline__ void store_first(double* out) const  // as (sum, compensation)
    {
        out[0] = (double)s.x / kScale;
        out[1] = ((double)c.x + (double)d.x) / kScale;
    }

private:
    __device__ __forceinline__ void add_sum(float s_, float c_, float d_, const Trig<float>& w)
    {
        add_product(V{s_, s_}, w);
        add_product(V{c_, c_}, w);
        d = __ffma2_rn(V{d_, d_}, w.hi, d);
    }
};
template <> struct Acc2<double> {
    using V = double2;
    static constexpr double kScale = 1.0;
    V s = {0.0, 0.0}, c = {0.0, 0.0};
    __device__ __forceinline__ void add(V v)
    {
        Comp a{s.x, c.x}, b{s.y, c.y};
        comp_add(a, v.x);
        comp_add(b, v.y);
        s = V{a.s, b.s};
        c = V{a.c, b.c};
    }
    __device__ __forceinline__ void add_product(V v, const Trig<double>& w) { add(V{v.x * w.hi.x, v.y * w.hi.y}); }
    __device__ __forceinline__ void add_first(const Acc2& a, const Trig<double>& w) { add_sum(a.s.x, a.c.x, w); }
    __device__ __forceinline__ void add_second(const Acc2& a, const Trig<double>& w) { add_sum(a.s.y, a.c.y, w); }
    __device__ __forceinline__ void merge(const Acc2& a)
    {
        add(a.s);
        c.x += a.c.x;
        c.y += a.c.y;
    }
    template <typename Fn>
    static __device__ __forceinline__ Acc2 of(const Acc2& a, const Acc2& b, Fn fn)
    {
        Acc2 r;
        r.s = fn(a.s, b.s);
        r.c = fn(a.c, b.c);
        return r;
    }
    __device__ __forceinline__ void store_first(double* out) const
    {
        out[0] = s.x;
        out[1] = c.x;
    }

private:
    __device__ __forceinline__ void add_sum(double s_, double c_, const Trig<double>& w)
    {
        const V q{s_ * w.hi.x, s_ * w.hi.y};
        add(q);
        c.x += fma(c_, w.hi.x, fma(s_, w.hi.x, -q.x));
        c.y += fma(c_, w.hi.y, fma(s_, w.hi.y, -q.y));
    }
};
// a lane's value v of the lane across bit o
template <typename V>
__device__ __forceinline__ V lane_across(V v, int o)
{
    return V{__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o)};
}
// Half of a warp's 2 N sums to either of the lanes across bit o: the first sums
// of the pairs where the bit is 0, the second ones where it is 1, packed in pairs
// again.  A reduction by halves moves and merges each sum once a level over all
// lanes: 36 shuffles and 8 merges for ten sums of three parts, not 150 and 25.
template <typename T, int N>
__device__ __forceinline__ void warp_halve(const Acc2<T> (&a)[N], Acc2<T> (&out)[(N + 1) / 2], int o)
{
    using V = typename Acc2<T>::V;
    const bool upper = (threadIdx.x & o) != 0;
    auto pack = [](const Acc2<T>& p, const Acc2<T>& q, bool second) {
        return Acc2<T>::of(p, q, [&](V u, V v) { return V{second ? u.y : u.x, second ? v.y : v.x}; });
    };
#pragma unroll
    for (int j = 0; j < (N + 1) / 2; ++j) {
        const Acc2<T> q = 2 * j + 1 < N ? a[2 * j + 1 < N ? 2 * j + 1 : 0] : Acc2<T>();
        const Acc2<T> give = pack(a[2 * j], q, !upper);
        out[j] = pack(a[2 * j], q, upper);
        out[j].merge(Acc2<T>::of(give, give, [&](V u, V) { return lane_across(u, o); }));
    }
}
// The warp's totals of five pairs of sums: the first sum of the result is that
// of pair `index` / 2, its second one where index is odd; index >= 10: nothing.
template <typename T>
__device__ __forceinline__ Acc2<T> warp_totals(const Acc2<T> (&a)[5], int& index)
{
    using V = typename Acc2<T>::V;
    Acc2<T> b[3], c[2], d[1], e[1];
    warp_halve(a, b, 16);
    warp_halve(b, c, 8);
    warp_halve(c, d, 4);
    warp_halve(d, e, 2);
    e[0].merge(Acc2<T>::of(e[0], e[0], [](V u, V) { return lane_across(u, 1); }));
    const int l = threadIdx.x;
    index = 2 * (2 * (2 * (l >> 1 & 1) + (l >> 2 & 1)) + (l >> 3 & 1)) + (l >> 4 & 1);
    return e[0];
}

template <typename T>
__global__ void k_diag_table(const BatchDomain<T>* __restrict__ doms, Trig<T>* table, int stride)
{
    const Geom G = doms[blockIdx.y].G;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= G.nx + G.ny) return;
    double s, c;
    sincospi(i < G.nx ? 2.0 * i / G.nx : 2.0 * (i - G.nx) / G.ny, &s, &c);
    Trig<T> e;
    e.set(c, s);
    table[(long long)blockIdx.y * stride + i] = e;
}

// Film diagnostics of domain blockIdx.y of a table (compensated sums):
// [0] h over the lattice; over the wetted nodes (h > h_wet) [1] h,
// [2] j_x, [3] j_y, [4] 1, [5] h cos(2 pi x / nx), [6] h sin(2 pi x / nx),
// [7] h cos(2 pi y / ny), [8] h sin(2 pi y / ny); over the lattice
// [9] h cos(phi), [10] h sin(phi) with phi = 2 pi (mx x / nx + my y / ny);
// and the largest h.  Block b writes kDiagPartial doubles at
// partials[(domain * gridDim.x + b) * kDiagPartial].
//
// A warp takes units of 32 columns x `rows` rows; a lane sums its own column
// down the rows, so the column's trigonometric factors multiply one sum per
// unit and the mode's phase splits into a row factor per node (none where the
// mode has no wave along y) and a column factor per unit (cos(a + b) from the
// two angles).  The unit height gives every warp of the launch one unit where it
// can, but at least kDiagRows rows (a unit's products and its reduction over the
// warp cost about five rows).
// Bound by the chains of TwoSums (60 paired operations a node, 90 with a row
// phase) and the latency of a row's nine loads: 32 warps an SM hide them better
// than 24 with the next row's loads in flight (32 domains, 7.6 M nodes, with the
// final kernel and the launches: 107 us; 24 warps 114; 40 spill: 124; skipping the
// wetted sums of dry rows by a vote 128).  In doubles 2150 us.
constexpr int kDiagPartial = 2 * kDiagSums + 1;
constexpr int kDiagRows = 16;
template <typename T, typename SM>
__global__ void __launch_bounds__(kMassThreads, sizeof(T) == 4 ? 4 : 1)
k_diag_partial(const BatchDomain<T>* __restrict__ doms, int parity, const Trig<T>* __restrict__ table, int stride,
               double h_wet, int mx, int my, double* partials)
{
    constexpr int NW = kMassThreads / 32;
    const BatchDomain<T>& D = doms[blockIdx.y];
    const Pops<T, SM> P = pops_of<T, SM>(D, parity);
    const Geom G = D.G;
    const Trig<T>* tx = table + (long long)blockIdx.y * stride;
    const Trig<T>* ty = tx + G.nx;
    using V = typename Acc2<T>::V;
    // per warp: (h, wetted h), (j_x, j_y), wetted h (cos, sin) of the column
    // and of the row angle, h (cos, sin) of the mode; wetted nodes; largest h
    __shared__ Acc2<T> sm[10][NW];  // first sums only
    __shared__ long long scount[NW];
    __shared__ T smax[NW];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane < 10) sm[lane][wid] = Acc2<T>();
    if (lane == 10) scount[wid] = 0;
    if (lane == 11) smax[wid] = -INFINITY;
    __syncwarp();
    // integer wave numbers reduced modulo the lattice, so phases stay exact
    const int kx = ((mx % G.nx) + G.nx) % G.nx, ky = ((my % G.ny) + G.ny) % G.ny;
    // hh > h_wet in the compute type: the nearest float at or below h_wet
    // separates the same heights
    T wet_above;
    if constexpr (std::is_same<T, float>::value) wet_above = __double2float_rd(h_wet);
    else wet_above = h_wet;
    const int warps = gridDim.x * NW;
    const int ux = (G.nx + 31) / 32, most = max(1, warps / ux);
    const int rows = max(kDiagRows, (G.ny + most - 1) / most), uy = (G.ny + rows - 1) / rows;
    for (int u = blockIdx.x * NW + wid; u < ux * uy; u += warps) {
        const int x = (u % ux) * 32 + lane, y0 = (u / ux) * rows, y1 = min(y0 + rows, G.ny);
        // over this column: (h, wetted h), wetted (j_x, j_y), wetted h (cos,
        // sin) of the row angle, h (cos, sin) of the row's mode phase
        Acc2<T> ah, aj, ar, am;
        int iy = (int)((long long)ky * y0 % G.ny), count = 0;
        T top = -INFINITY;
        if (x < G.nx) {
            const int xm = wrapi(x - 1, G.nx), xp = wrapi(x + 1, G.nx);
            int ra = wrapi(y0 - 1, G.ny) * P.pitch, r0 = y0 * P.pitch;  // rows y - 1, y
            auto pull = [&](int y, T(&v)[9]) {  // row y, whose neighbours are ra and the one after r0
                const int rb = y + 1 == G.ny ? 0 : r0 + P.pitch;
                v[0] = P.full(0, r0 + x);
                v[1] = P.full(1, r0 + xm);
                v[2] = P.full(2, ra + xm);
                v[3] = P.full(3, ra + x);
                v[4] = P.full(4, ra + xp);
                v[5] = P.full(5, r0 + xp);
                v[6] = P.full(6, rb + xp);
                v[7] = P.full(7, rb + x);
                v[8] = P.full(8, rb + xm);
                ra = r0;
                r0 = rb;
            };
            for (int y = y0; y < y1; ++y) {
                T v[9];
                pull(y, v);
                T hh, jx, jy;
                moments9(v, hh, jx, jy);
                const bool wet = hh > wet_above;
                const T hw = wet ? hh : T(0);
                const Trig<T> w = ty[y];
                const T k = T(Acc2<T>::kScale), hs = hh * k, ws = hw * k;
                ah.add(V{hs, ws});
                aj.add(V{wet ? jx * k : T(0), wet ? jy * k : T(0)});
                ar.add_product(V{ws, ws}, w);
                if (ky != 0) am.add_product(V{hs, hs}, ty[iy]);
                count += wet;
                iy += ky;
                if (iy >= G.ny) iy -= G.ny;
                top = fmax(top, hh);
            }
        }
        const int xc = min(x, G.nx - 1);  // a lane past the lattice holds zeros
        const Trig<T> w = tx[xc], m = tx[(long long)kx * xc % G.nx];
        Acc2<T> ac, ap;  // the column angle; the mode: cos(a + b), sin(a + b)
        ac.add_second(ah, w);
        if (ky == 0) {  // the rows' phase is 0: (1, 0) times the sum of h
            ap.add_first(ah, m);
        } else {
            ap.add_first(am, m);
            ap.add_second(am, m.turned());
        }
        int k;
        const Acc2<T> q = warp_totals<T>({ah, aj, ac, ar, ap}, k);
        if (k < 10 && lane % 2 == 0) sm[k][wid].merge(q);
        count = __reduce_add_sync(0xffffffffu, count);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) top = fmax(top, __shfl_down_sync(0xffffffffu, top, o));
        if (lane == 0) {
            scount[wid] += count;
            smax[wid] = fmax(smax[wid], top);
        }
    }
    __syncthreads();
    double* out = partials + ((long long)blockIdx.y * gridDim.x + blockIdx.x) * kDiagPartial;
    const int k = threadIdx.x;
    if (k < 10) {
        Acc2<T> b = sm[k][0];
        for (int w = 1; w < NW; ++w) b.merge(sm[k][w]);
        b.store_first(out + 2 * (k < 4 ? k : k + 1));  // sums 0 .. 3, 5 .. 10
    } else if (k == 10) {
        long long b = 0;
        for (int w = 0; w < NW; ++w) b += scount[w];
        out[8] = (double)b;  // exact below 2^53
        out[9] = 0.0;
    } else if (k == 11) {
        T b = smax[0];
        for (int w = 1; w < NW; ++w) b = fmax(b, smax[w]);
        out[2 * kDiagSums] = b;
    }
}

// One warp per value: block (k, domain) reduces the partials of the domain's
// nb blocks into field k of out[domain * kDiagOut ..], the fields of
// tf_lbm_diag (sums 0..4, the maximum, sums 5..10).  A warp each, not a block
// per domain, so that the FP64 adds of the twelve values spread over SMs.
__global__ void __launch_bounds__(32) k_diag_final(const double* __restrict__ partials, int nb, double* out)
{
    const double* p = partials + (long long)blockIdx.y * nb * kDiagPartial;
    const int k = blockIdx.x;
    double r;
    if (k == 5) {
        double m = -INFINITY;
        for (int i = threadIdx.x; i < nb; i += 32) m = fmax(m, p[(long long)i * kDiagPartial + 2 * kDiagSums]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        r = m;
    } else {
        const int q = 2 * (k < 5 ? k : k - 1);
        Comp a{0.0, 0.0};
        for (int i = threadIdx.x; i < nb; i += 32) {
            comp_add(a, p[(long long)i * kDiagPartial + q]);
            a.c += p[(long long)i * kDiagPartial + q + 1];
        }
        a = warp_reduce(a);
        r = a.s + a.c;
    }
    if (threadIdx.x == 0) out[(long long)blockIdx.y * kDiagOut + k] = r;
}

// ---- term balance of the appendix (Eq. magnitude): fields h, j, p, div j
template <typename T, typename SM>
__global__ void k_tn_fields(Pops<T, SM> P, T* hb, T* jxb, T* jyb, Geom G)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= G.nx) return;
    T v[9], hh, jx, jy;
    pull_at(P, G, x, y, v);
    moments9(v, hh, jx, jy);
    const long long i = (long long)y * G.nx + x;
    hb[i] = hh;
    jxb[i] = jx;
    jyb[i] = jy;
}

// d/dx and d/dy of a field with the stencil of Eq. (derivative)
template <typename T>
struct Stencil {
    const T* f;
    Geom G;
    int x, y, xm, xp, ym, yp;
    __device__ Stencil(const T* f_, const Geom& G_, int x_, int y_) : f(f_), G(G_), x(x_), y(y_)
    {
        xm = wrapi(x - 1, G.nx);
        xp = wrapi(x + 1, G.nx);
        ym = wrapi(y - 1, G.ny);
        yp = wrapi(y + 1, G.ny);
    }
    __device__ T at(int yy, int xx) const { return f[(long long)yy * G.nx + xx]; }
    __device__ T dx() const
    {
        return (at(y, xp) - at(y, xm)) / T(3) + (at(yp, xp) - at(yp, xm) + at(ym, xp) - at(ym, xm)) / T(12);
    }
    __device__ T dy() const
    {
        return (at(yp, x) - at(ym, x)) / T(3) + (at(yp, xp) - at(ym, xp) + at(yp, xm) - at(ym, xm)) / T(12);
    }
    // Eq. (n_laplace) with the reading (1/6)[4 sum_axis + sum_diag - 20 phi]
    __device__ T lap() const
    {
        const T axis = at(y, xm) + at(y, xp) + at(ym, x) + at(yp, x);
        const T diag = at(ym, xm) + at(ym, xp) + at(yp, xm) + at(yp, xp);
        return (T(4) * axis + diag - T(20) * at(y, x)) / T(6);
    }
};

template <typename T>
__global__ void k_tn_div(const T* __restrict__ jx, const T* __restrict__ jy, T* div, Geom G)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= G.nx) return;
    div[(long long)y * G.nx + x] = Stencil<T>(jx, G, x, y).dx() + Stencil<T>(jy, G, x, y).dy();
}

// Sums of squares of the x-components of -h d_x p, -nu alpha(h) u_x and
// nu lap(j_x) + 2 nu d_x(div j) (three (s, c) pairs per block).
template <typename T>
__global__ void __launch_bounds__(kMassThreads) k_tn_terms(const T* __restrict__ hb, const T* __restrict__ jxb,
                                                           const T* __restrict__ pb, const T* __restrict__ db,
                                                           Geom G, Consts<T> C, double* partials)
{
    Comp a[3] = {{0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}};
    const long long n = (long long)G.nx * G.ny;
    const double nu = (double)C.nu6 / 6.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(i % G.nx), y = (int)(i / G.nx);
        const double h = (double)hb[i], jx = (double)jxb[i], d = (double)C.delta;
        const double tp = -h * (double)Stencil<T>(pb, G, x, y).dx();
        // nu alpha(h) u_x = 6 nu j_x / (2 h^2 + 6 delta h + 3 delta^2), Eqs. (forcefric, alphafric)
        const double tf = -6.0 * nu * jx / (2.0 * h * h + 6.0 * d * h + 3.0 * d * d);
        const double td = nu * (double)Stencil<T>(jxb, G, x, y).lap() + 2.0 * nu * (double)Stencil<T>(db, G, x, y).dx();
        comp_add(a[0], tp * tp);
        comp_add(a[1], tf * tf);
        comp_add(a[2], td * td);
    }
    for (int k = 0; k < 3; ++k) {
        const Comp b = block_sum(a[k]);
        if (threadIdx.x == 0) {
            partials[2 * (k * gridDim.x + blockIdx.x)] = b.s;
            partials[2 * (k * gridDim.x + blockIdx.x) + 1] = b.c;
        }
    }
}

__global__ void __launch_bounds__(kMassThreads) k_tn_final(const double* __restrict__ partials, int nb, double n,
                                                           double* out)
{
    for (int k = 0; k < 3; ++k) {
        Comp a{0.0, 0.0};
        for (int i = threadIdx.x; i < nb; i += blockDim.x) {
            comp_add(a, partials[2 * (k * nb + i)]);
            a.c += partials[2 * (k * nb + i) + 1];
        }
        const Comp b = block_sum(a);
        if (threadIdx.x == 0) out[k] = sqrt((b.s + b.c) / n);
    }
}

// Smallest of n values (NaNs ignored; +inf when there is none).
template <typename T>
__global__ void __launch_bounds__(kMassThreads) k_min_partial(const T* __restrict__ x, long long n,
                                                              double* partials)
{
    double m = -INFINITY;  // max of -x
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        m = fmax(m, -(double)x[i]);
    m = block_max(m);
    if (threadIdx.x == 0) partials[blockIdx.x] = m;
}

__global__ void __launch_bounds__(kMassThreads) k_min_final(const double* partials, int n, double* out)
{
    double m = -INFINITY;
    for (int i = threadIdx.x; i < n; i += blockDim.x) m = fmax(m, partials[i]);
    m = block_max(m);
    if (threadIdx.x == 0) *out = -m;
}

__global__ void __launch_bounds__(kMassThreads) k_mass_final(const double* partials, int n, double* out)
{
    Comp a{0.0, 0.0};
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        comp_add(a, partials[2 * i]);
        a.c += partials[2 * i + 1];
    }
    a = warp_reduce(a);
    __shared__ Comp sm[kMassThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) sm[wid] = a;
    __syncthreads();
    if (wid == 0) {
        Comp b = lane < kMassThreads / 32 ? sm[lane] : Comp{0.0, 0.0};
        b = warp_reduce(b);
        if (lane == 0) *out = b.s + b.c;
    }
}

template <typename T, typename SM>
__global__ void k_check(Pops<T, SM> P, Geom G, int* flag)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    int bad = 0;
    if (x < G.nx) {
        T v[9], hh, jx, jy;
        pull_at(P, G, x, y, v);
        for (int l = 0; l < 9; ++l)
            if (!isfinite((double)v[l])) bad |= 1;
        moments9(v, hh, jx, jy);
        if (!isfinite((double)hh)) bad |= 1;
        else if (!(hh > T(0))) bad |= 2;
    }
    bad = __reduce_or_sync(0xffffffffu, bad);
    if (bad && (threadIdx.x & 31) == 0) atomicOr(flag, bad);
}

// float to double and back, with the bits FP64 conversions give.  The FP64
// pipe takes 16 clocks a warp instruction; nine conversions a node bounded the
// state import and export (2^20 nodes: 24 and 27 us a pass, 16 us now), so the
// exponent is moved by integer instructions where a node's nine values are
// normal or zero; other nodes take the conversions.
__device__ __forceinline__ bool widens(float v)  // normal or zero
{
    const uint32_t m = __float_as_uint(v) & 0x7fffffffu;
    return m - 0x00800000u < 0x7f000000u || m == 0;
}
__device__ __forceinline__ double widen(float v)
{
    const uint32_t u = __float_as_uint(v), m = u & 0x7fffffffu;
    return __hiloint2double((int)((u & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u)), (int)(u << 29));
}
__device__ __forceinline__ bool narrows(double v)  // [2^-126, 2^127): the rounding cannot overflow; or zero
{
    const uint32_t m = (uint32_t)__double2hiint(v) & 0x7fffffffu;
    return m - 0x38100000u < 0x0fd00000u || (m | (uint32_t)__double2loint(v)) == 0;
}
__device__ __forceinline__ float narrow(double v)
{
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v), m = hi & 0x7fffffffu;
    uint32_t r = ((m - 0x38000000u) << 3) | (lo >> 29);
    const uint32_t rest = lo & 0x1fffffffu;
    r += rest > 0x10000000u || (rest == 0x10000000u && (r & 1u));  // to nearest, ties to even
    return __uint_as_float((hi & 0x80000000u) | ((m | lo) == 0 ? 0u : r));
}

// State export in double: decoded values plus href in double are exact for
// float and 16-bit storage, so an export / import round trip reproduces the
// stored bits.
template <typename T, typename SM>
__global__ void k_get_state(Pops<T, SM> P, double* out, Geom G)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= G.nx) return;
    const long long n = (long long)G.nx * G.ny, i = (long long)y * G.nx + x;
    const Around N(x, y, G.nx, G.ny, P.pitch);
    T v[9];
#pragma unroll
    for (int l = 0; l < 9; ++l) v[l] = P.raw(l, N.at(-cx_of(l), -cy_of(l)));
    double d[9];
    if constexpr (std::is_same<T, float>::value) {
        bool plain = true;
#pragma unroll
        for (int l = 0; l < 9; ++l) plain = plain && widens(v[l]);
        if (plain) {
#pragma unroll
            for (int l = 0; l < 9; ++l) d[l] = widen(v[l]);
        } else {
#pragma unroll
            for (int l = 0; l < 9; ++l) d[l] = (double)v[l];
        }
    } else {
#pragma unroll
        for (int l = 0; l < 9; ++l) d[l] = v[l];
    }
    d[0] += (double)P.href;
#pragma unroll
    for (int l = 0; l < 9; ++l) out[l * n + i] = d[l];
}

// Post-streaming populations in the compute type, [9][ny][nx] (adjoint input).
template <typename T, typename SM>
__global__ void k_export_state(Pops<T, SM> P, T* out, Geom G)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= G.nx) return;
    T v[9];
    pull_at(P, G, x, y, v);
    const long long n = (long long)G.nx * G.ny, i = (long long)y * G.nx + x;
#pragma unroll
    for (int l = 0; l < 9; ++l) out[l * n + i] = v[l];
}

template <typename T, typename SM>
__global__ void k_set_state(Pops<T, SM> P, const double* __restrict__ in, Geom G)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= G.nx) return;
    const long long n = (long long)G.nx * G.ny;
    const Around N(x, y, G.nx, G.ny, G.nx);
    double d[9];
#pragma unroll
    for (int l = 0; l < 9; ++l) d[l] = in[l * n + N.at(cx_of(l), cy_of(l))];
    d[0] -= (double)P.href;
    T v[9];
    if constexpr (std::is_same<T, float>::value) {
        bool plain = true;
#pragma unroll
        for (int l = 0; l < 9; ++l) plain = plain && narrows(d[l]);
        if (plain) {
#pragma unroll
            for (int l = 0; l < 9; ++l) v[l] = narrow(d[l]);
        } else {
#pragma unroll
            for (int l = 0; l < 9; ++l) v[l] = (float)d[l];
        }
    } else {
#pragma unroll
        for (int l = 0; l < 9; ++l) v[l] = d[l];
    }
    const int o = P.at(y, x);
#pragma unroll
    for (int l = 0; l < 9; ++l) P.put(l, o, v[l]);
}

inline dim3 grid2d(const Geom& G, int bx) { return dim3((G.nx + bx - 1) / bx, G.ny); }

template <typename T, typename SM>
cudaError_t init_t(const StoreDesc& D, void* f, const void* h0, const Geom& G, double g, cudaStream_t st)
{
    k_init<T, SM><<<grid2d(G, 128), 128, 0, st>>>(make_pops<T, SM>(f, G, D), (const T*)h0, G, T(g));
    return cudaGetLastError();
}

template <typename T, typename SM>
cudaError_t moments_t(const StoreDesc& D, const void* f, void* h, void* ux, void* uy, const Geom& G,
                      cudaStream_t st)
{
    k_moments<T, SM><<<grid2d(G, 128), 128, 0, st>>>(make_pops<T, SM>(f, G, D), (T*)h, (T*)ux, (T*)uy, G);
    return cudaGetLastError();
}

template <typename T, typename SM>
cudaError_t pf_t(const StoreDesc& D, const void* f, const void* kappa, void* p, void* fx, void* fy,
                 const Geom& G, const Consts<T>& C, cudaStream_t st)
{
    auto launch = [&](auto rows) {
        constexpr int Y = decltype(rows)::value;
        const dim3 grid((G.nx + kPfX - 1) / kPfX, (G.ny + Y - 1) / Y);
        k_pf<T, SM, Y><<<grid, kPfThreads, 0, st>>>(make_pops<T, SM>(f, G, D), (const T*)kappa, (T*)p, (T*)fx, (T*)fy, G, C);
        return cudaGetLastError();
    };
    if constexpr (sizeof(T) == 8) {
        if (2LL * ((G.nx + kPfX - 1) / kPfX) * ((G.ny + 15) / 16) < sm_count()) return launch(std::integral_constant<int, 4>());
    }
    return launch(std::integral_constant<int, 16>());
}

template <typename T, typename SM>
cudaError_t mass_t(const StoreDesc& D, const void* f, const Geom& G, double* partials, int nblocks,
                   double* result, cudaStream_t st)
{
    k_mass_partial<T, SM><<<nblocks, kMassThreads, 0, st>>>(make_pops<T, SM>(f, G, D), G, partials);
    k_mass_final<<<1, kMassThreads, 0, st>>>(partials, nblocks, result);
    return cudaGetLastError();
}

template <typename T, typename SM>
cudaError_t diag_t(const void* doms, int ndom, int parity, const void* table, int stride, double h_wet, int mx,
                   int my, double* partials, int nb, double* out, cudaStream_t st)
{
    k_diag_partial<T, SM><<<dim3(nb, ndom), kMassThreads, 0, st>>>((const BatchDomain<T>*)doms, parity,
                                                                  (const Trig<T>*)table, stride, h_wet, mx, my, partials);
    k_diag_final<<<dim3(kDiagOut, ndom), 32, 0, st>>>(partials, nb, out);
    return cudaGetLastError();
}

template <typename T, typename SM>
cudaError_t term_norms_t(const StoreDesc& D, const void* f, const void* kappa, const Geom& G, const Consts<T>& C,
                         void* scratch, double* partials, int nb, double* out, cudaStream_t st)
{
    const long long n = (long long)G.nx * G.ny;
    T* hb = (T*)scratch;
    T* jxb = hb + n;
    T* jyb = jxb + n;
    T* pb = jyb + n;
    T* db = pb + n;
    k_tn_fields<T, SM><<<grid2d(G, 128), 128, 0, st>>>(make_pops<T, SM>(f, G, D), hb, jxb, jyb, G);
    k_pf_p<T><<<grid2d(G, 128), 128, 0, st>>>(hb, (const T*)kappa, pb, G, C);
    k_tn_div<T><<<grid2d(G, 128), 128, 0, st>>>(jxb, jyb, db, G);
    k_tn_terms<T><<<nb, kMassThreads, 0, st>>>(hb, jxb, pb, db, G, C, partials);
    k_tn_final<<<1, kMassThreads, 0, st>>>(partials, nb, (double)n, out);
    return cudaGetLastError();
}

template <typename T, typename SM>
cudaError_t check_t(const StoreDesc& D, const void* f, const Geom& G, int* flag, cudaStream_t st)
{
    k_check<T, SM><<<grid2d(G, 128), 128, 0, st>>>(make_pops<T, SM>(f, G, D), G, flag);
    return cudaGetLastError();
}

template <typename T, typename SM>
cudaError_t get_t(const StoreDesc& D, const void* f, double* out, const Geom& G, cudaStream_t st)
{
    k_get_state<T, SM><<<grid2d(G, 128), 128, 0, st>>>(make_pops<T, SM>(f, G, D), out, G);
    return cudaGetLastError();
}

template <typename T, typename SM>
cudaError_t export_t(const StoreDesc& D, const void* f, void* out, const Geom& G, cudaStream_t st)
{
    k_export_state<T, SM><<<grid2d(G, 128), 128, 0, st>>>(make_pops<T, SM>(f, G, D), (T*)out, G);
    return cudaGetLastError();
}

template <typename T, typename SM>
cudaError_t set_t(const StoreDesc& D, void* f, const double* in, const Geom& G, cudaStream_t st)
{
    k_set_state<T, SM><<<grid2d(G, 128), 128, 0, st>>>(make_pops<T, SM>(f, G, D), in, G);
    return cudaGetLastError();
}

}  // namespace

int mass_blocks(const Geom& G)
{
    long long rows = 9LL * G.ny;
    return (int)(rows < 1184 ? rows : 1184);
}

// Dispatch over the storage type: F32 and the 16-bit stores compute in float,
// F64 in double.
#define TFLBM_DISPATCH(D, CALL)                                                      \
    switch ((D).store) {                                                             \
        case kStoreF32: { using T = float; using SM = float; return CALL; }          \
        case kStoreF64: { using T = double; using SM = double; return CALL; }        \
        case kStoreF16: { using T = float; using SM = __half; return CALL; }         \
        case kStoreBF16: { using T = float; using SM = __nv_bfloat16; return CALL; } \
        default: return cudaErrorInvalidValue;                                       \
    }

cudaError_t aux_init(const StoreDesc& D, void* f, const void* h0, const Geom& G, double g, cudaStream_t st)
{
    TFLBM_DISPATCH(D, (init_t<T, SM>(D, f, h0, G, g, st)))
}

cudaError_t aux_moments(const StoreDesc& D, const void* f, void* h, void* ux, void* uy, const Geom& G,
                        cudaStream_t st)
{
    TFLBM_DISPATCH(D, (moments_t<T, SM>(D, f, h, ux, uy, G, st)))
}

cudaError_t aux_pressure_force(const StoreDesc& D, const void* f, const void* kappa, void* p, void* fx,
                               void* fy, const Geom& G, const Consts<float>* C32, const Consts<double>* C64,
                               cudaStream_t st)
{
    switch (D.store) {
        case kStoreF32: return pf_t<float, float>(D, f, kappa, p, fx, fy, G, *C32, st);
        case kStoreF64: return pf_t<double, double>(D, f, kappa, p, fx, fy, G, *C64, st);
        case kStoreF16: return pf_t<float, __half>(D, f, kappa, p, fx, fy, G, *C32, st);
        case kStoreBF16: return pf_t<float, __nv_bfloat16>(D, f, kappa, p, fx, fy, G, *C32, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t aux_mass(const StoreDesc& D, const void* f, const Geom& G, double* partials, int nblocks,
                     double* result, cudaStream_t st)
{
    TFLBM_DISPATCH(D, (mass_t<T, SM>(D, f, G, partials, nblocks, result, st)))
}

cudaError_t aux_diag_table(bool dbl, const void* doms, int ndom, int stride, void* table, cudaStream_t st)
{
    const dim3 grid((stride + 255) / 256, ndom);
    if (dbl) k_diag_table<double><<<grid, 256, 0, st>>>((const BatchDomain<double>*)doms, (Trig<double>*)table, stride);
    else k_diag_table<float><<<grid, 256, 0, st>>>((const BatchDomain<float>*)doms, (Trig<float>*)table, stride);
    return cudaGetLastError();
}

cudaError_t aux_diag(int store, const void* doms, int ndom, int parity, const void* table, int stride, double h_wet,
                     int mx, int my, double* partials, int nb, double* out, cudaStream_t st)
{
    switch (store) {
        case kStoreF32: return diag_t<float, float>(doms, ndom, parity, table, stride, h_wet, mx, my, partials, nb, out, st);
        case kStoreF64: return diag_t<double, double>(doms, ndom, parity, table, stride, h_wet, mx, my, partials, nb, out, st);
        case kStoreF16: return diag_t<float, __half>(doms, ndom, parity, table, stride, h_wet, mx, my, partials, nb, out, st);
        case kStoreBF16:
            return diag_t<float, __nv_bfloat16>(doms, ndom, parity, table, stride, h_wet, mx, my, partials, nb, out, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t aux_term_norms(const StoreDesc& D, const void* f, const void* kappa, const Geom& G,
                           const Consts<float>* C32, const Consts<double>* C64, void* scratch, double* partials,
                           int nb, double* out, cudaStream_t st)
{
    switch (D.store) {
        case kStoreF32: return term_norms_t<float, float>(D, f, kappa, G, *C32, scratch, partials, nb, out, st);
        case kStoreF64: return term_norms_t<double, double>(D, f, kappa, G, *C64, scratch, partials, nb, out, st);
        case kStoreF16: return term_norms_t<float, __half>(D, f, kappa, G, *C32, scratch, partials, nb, out, st);
        case kStoreBF16:
            return term_norms_t<float, __nv_bfloat16>(D, f, kappa, G, *C32, scratch, partials, nb, out, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t aux_check(const StoreDesc& D, const void* f, const Geom& G, int* flag, cudaStream_t st)
{
    TFLBM_DISPATCH(D, (check_t<T, SM>(D, f, G, flag, st)))
}

cudaError_t aux_get_state(const StoreDesc& D, const void* f, double* out, const Geom& G, cudaStream_t st)
{
    TFLBM_DISPATCH(D, (get_t<T, SM>(D, f, out, G, st)))
}

cudaError_t aux_export_state(const StoreDesc& D, const void* f, void* out, const Geom& G, cudaStream_t st)
{
    TFLBM_DISPATCH(D, (export_t<T, SM>(D, f, out, G, st)))
}

cudaError_t aux_set_state(const StoreDesc& D, void* f, const double* in, const Geom& G, cudaStream_t st)
{
    TFLBM_DISPATCH(D, (set_t<T, SM>(D, f, in, G, st)))
}

cudaError_t aux_kappa(bool dbl, void* kappa, const void* theta, int nx, int ny, int ne, int me,
                      double hstar, cudaStream_t st)
{
    const long long n = (long long)nx * ny;
    const int blocks = (int)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096);
    if (dbl) k_kappa<double><<<blocks, 256, 0, st>>>((double*)kappa, (const double*)theta, n, ne, me, hstar);
    else k_kappa<float><<<blocks, 256, 0, st>>>((float*)kappa, (const float*)theta, n, ne, me, hstar);
    return cudaGetLastError();
}

cudaError_t aux_min(bool dbl, const void* x, long long n, double* partials, int nblocks, double* result,
                    cudaStream_t st)
{
    if (dbl) k_min_partial<double><<<nblocks, kMassThreads, 0, st>>>((const double*)x, n, partials);
    else k_min_partial<float><<<nblocks, kMassThreads, 0, st>>>((const float*)x, n, partials);
    k_min_final<<<1, kMassThreads, 0, st>>>(partials, nblocks, result);
    return cudaGetLastError();
}


}  // namespace tflbm
