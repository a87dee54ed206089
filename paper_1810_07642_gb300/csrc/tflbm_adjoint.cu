// Discrete adjoint of the thin-film step and the checkpointed gradient tape.
//
// State: the post-streaming populations f(t), [9][ny][nx] in the compute
// type.  One step is f(t+1) = S(C(f(t))) with C the forced BGK collision of
// Eq. (LBE), using the force of Eq. (force) and the film pressure of
// Eqs. (pfilm, disjoiningP), and S the streaming.  Given a(t+1) = dL/df(t+1),
// the adjoint step returns a(t) = (d S C / d f(t))^T a(t+1) and adds
// (d S C / d kappa)^T a(t+1) to dL/dkappa.  Derivation, phase by phase
// (E_l are the equilibria of Eq. (equilibria) written in h and j = h u):
//   mu_l(x)  = a_l(x + c_l, t+1)                          streaming^T
//   aF       = sum_l 3 w_l c_l mu_l,  aE_l = omega mu_l    collision^T
//   aH       = sum_l aE_l dE_l/dh + aF.(G - grad p) - fr'(h) aF.j
//   aJ       = sum_l aE_l dE_l/dj - fr(h) aF,  ag = -h aF  force^T
//   ap(y)    = sum_l 3 w_l c_l . ag(y - c_l)               Eq. (derivative)^T
//   aPi = -gamma s ap: dL/dkappa += aPi (r^n - r^m), aH += aPi kappa (m r^m - n r^n)/h
//   aH      += lap(-gamma ap)                              Eq. (n_laplace) is symmetric
//   a_l(x,t) = aH + c_l . aJ + (1 - omega) mu_l            moments^T
// with r = h_*/h, fr = 6 nu / (2h^2 + 6 delta h + 3 delta^2).
//
// The gradient tape runs the forward from the handle's state in tile steps
// that record h and j of every state they start from (all that the adjoint
// needs of f, see tflbm_adjoint_tile.cuh).  Where the records of all steps fit
// in kTapeBytes it keeps them; else it keeps a copy of the state every K steps
// (K ~ sqrt(T)) and the backward pass recomputes each segment's records from
// its copy, in reverse order of the segments.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <vector>

#include "tflbm_adjoint_tile.cuh"
#include "tflbm_handle.h"

namespace tflbm {
namespace {

__device__ __constant__ int aCx[9] = {0, 1, 1, 0, -1, -1, -1, 0, 1};
__device__ __constant__ int aCy[9] = {0, 0, 1, 1, 1, 0, -1, -1, -1};


template <typename T> __device__ __forceinline__ T wgt(int l) { return l == 0 ? T(4.0 / 9.0) : ((l & 1) ? T(1.0 / 9.0) : T(1.0 / 36.0)); }

struct Dims {
    int nx, ny;
    long long n;  // nx * ny
};

// Wrapped neighbourhood of node (x, y): row offsets of y-1, y, y+1 and
// columns x-1, x, x+1 (no integer division).
struct Nbr {
    long long r[3];
    int c[3];
    __device__ __forceinline__ Nbr(int x, int y, const Dims& D)
    {
        r[0] = (long long)(y == 0 ? D.ny - 1 : y - 1) * D.nx;
        r[1] = (long long)y * D.nx;
        r[2] = (long long)(y + 1 == D.ny ? 0 : y + 1) * D.nx;
        c[0] = x == 0 ? D.nx - 1 : x - 1;
        c[1] = x;
        c[2] = x + 1 == D.nx ? 0 : x + 1;
    }
    // index of node (x + dx, y + dy), dx, dy in {-1, 0, 1}
    __device__ __forceinline__ long long at(int dy, int dx) const { return r[dy + 1] + c[dx + 1]; }
};

// h, j of the state f at every node
template <typename T>
__global__ void k_adj_moments(const T* __restrict__ f, T* h, T* jx, T* jy, Dims D)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= D.nx) return;
    const long long i = (long long)y * D.nx + x;
    T s = 0, sx = 0, sy = 0;
#pragma unroll
    for (int l = 0; l < 9; ++l) {
        const T v = f[l * D.n + i];
        s += v;
        sx += T(aCx[l]) * v;
        sy += T(aCy[l]) * v;
    }
    h[i] = s;
    jx[i] = sx;
    jy[i] = sy;
}

// film pressure p = -gamma (lap h + s kappa (r^n - r^m))
template <typename T>
__global__ void k_adj_pressure(const T* __restrict__ h, const T* __restrict__ kappa, T* p, Dims D,
                               Consts<T> C)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= D.nx) return;
    const Nbr nb(x, y, D);
    auto H = [&](int dy, int dx) { return h[nb.at(dy, dx)]; };
    const T axis = H(0, -1) + H(0, 1) + H(-1, 0) + H(1, 0);
    const T diag = H(-1, -1) + H(-1, 1) + H(1, -1) + H(1, 1);
    const T hh = H(0, 0);
    T lap = (T(4) * axis + diag - T(20) * hh) / T(6);
    const long long i = (long long)y * D.nx + x;
    const T kap = kappa ? kappa[i] : C.kappa_u;
    const T r = C.hstar / hh;
    T rn = 1, rm = 1;
    for (int k = 0; k < C.n_exp; ++k) rn *= r;
    for (int k = 0; k < C.m_exp; ++k) rm *= r;
    p[i] = -C.gamma * (lap + C.pi_sgn * kap * (rn - rm));
}

// collision and force adjoint at every node
template <typename T>
__global__ void k_adj_collide(const T* __restrict__ h, const T* __restrict__ jx, const T* __restrict__ jy,
                              const T* __restrict__ p, const T* __restrict__ a_next, T* aH, T* aJx,
                              T* aJy, T* agx, T* agy, Dims D, Consts<T> C)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= D.nx) return;
    const long long i = (long long)y * D.nx + x;
    const Nbr nb(x, y, D);
    auto Pp = [&](int dy, int dx) { return p[nb.at(dy, dx)]; };
    // Eq. (derivative) at the node
    const T gpx = (Pp(0, 1) - Pp(0, -1)) / T(3) + (Pp(1, 1) - Pp(1, -1) + Pp(-1, 1) - Pp(-1, -1)) / T(12);
    const T gpy = (Pp(1, 0) - Pp(-1, 0)) / T(3) + (Pp(1, 1) - Pp(-1, 1) + Pp(1, -1) - Pp(-1, -1)) / T(12);
    const T hh = h[i], Jx = jx[i], Jy = jy[i], j2 = Jx * Jx + Jy * Jy, g = C.g, w = C.omega;
    T aFx = 0, aFy = 0, ah = 0, ajx = 0, ajy = 0;
#pragma unroll
    for (int l = 0; l < 9; ++l) {
        const T m = a_next[l * D.n + nb.at(aCy[l], aCx[l])];
        aFx += T(3) * wgt<T>(l) * T(aCx[l]) * m;
        aFy += T(3) * wgt<T>(l) * T(aCy[l]) * m;
        const T am = w * m;
        const T cj = T(aCx[l]) * Jx + T(aCy[l]) * Jy;
        T dh, djx, djy;
        if (l == 0) {
            dh = T(1) - T(5) * g * hh / T(3) + T(2) * j2 / (T(3) * hh * hh);
            djx = -T(4) * Jx / (T(3) * hh);
            djy = -T(4) * Jy / (T(3) * hh);
        } else if (l & 1) {
            dh = g * hh / T(3) - cj * cj / (T(2) * hh * hh) + j2 / (T(6) * hh * hh);
            djx = T(aCx[l]) / T(3) + cj * T(aCx[l]) / hh - Jx / (T(3) * hh);
            djy = T(aCy[l]) / T(3) + cj * T(aCy[l]) / hh - Jy / (T(3) * hh);
        } else {
            dh = g * hh / T(12) - cj * cj / (T(8) * hh * hh) + j2 / (T(24) * hh * hh);
            djx = T(aCx[l]) / T(12) + cj * T(aCx[l]) / (T(4) * hh) - Jx / (T(12) * hh);
            djy = T(aCy[l]) / T(12) + cj * T(aCy[l]) / (T(4) * hh) - Jy / (T(12) * hh);
        }
        ah += am * dh;
        ajx += am * djx;
        ajy += am * djy;
    }
    const T den = T(2) * hh * hh + C.delta * (T(6) * hh + T(3) * C.delta);
    const T nu6 = C.nu6;
    const T fr = nu6 / den;
    const T dfr = -nu6 * (T(4) * hh + T(6) * C.delta) / (den * den);
    ah += aFx * (C.gx - gpx) + aFy * (C.gy - gpy) - dfr * (aFx * Jx + aFy * Jy);
    aH[i] = ah;
    aJx[i] = ajx - fr * aFx;
    aJy[i] = ajy - fr * aFy;
    agx[i] = -hh * aFx;
    agy[i] = -hh * aFy;
}

// transpose of the gradient stencil, then the film-pressure adjoint
template <typename T>
__global__ void k_adj_pressure_t(const T* __restrict__ agx, const T* __restrict__ agy,
                                 const T* __restrict__ h, const T* __restrict__ kappa, T* aH, T* alap,
                                 T* grad_kappa, Dims D, Consts<T> C)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= D.nx) return;
    const long long i = (long long)y * D.nx + x;
    const Nbr nb(x, y, D);
    T ap = 0;
#pragma unroll
    for (int l = 0; l < 9; ++l) {
        const long long k = nb.at(-aCy[l], -aCx[l]);
        ap += T(3) * wgt<T>(l) * (T(aCx[l]) * agx[k] + T(aCy[l]) * agy[k]);
    }
    alap[i] = -C.gamma * ap;
    const T api = -C.gamma * C.pi_sgn * ap;
    const T hh = h[i];
    const T r = C.hstar / hh;
    T rn = 1, rm = 1;
    for (int k = 0; k < C.n_exp; ++k) rn *= r;
    for (int k = 0; k < C.m_exp; ++k) rm *= r;
    const T kap = kappa ? kappa[i] : C.kappa_u;
    grad_kappa[i] += api * (rn - rm);
    aH[i] += api * kap * (T(C.m_exp) * rm - T(C.n_exp) * rn) / hh;
}

// Laplacian (symmetric) and the moments' transpose
template <typename T>
__global__ void k_adj_out(const T* __restrict__ aH, const T* __restrict__ alap, const T* __restrict__ aJx,
                          const T* __restrict__ aJy, const T* __restrict__ a_next, T* a, Dims D,
                          Consts<T> C)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= D.nx) return;
    const long long i = (long long)y * D.nx + x;
    const Nbr nb(x, y, D);
    auto Ls = [&](int dy, int dx) { return alap[nb.at(dy, dx)]; };
    const T axis = Ls(0, -1) + Ls(0, 1) + Ls(-1, 0) + Ls(1, 0);
    const T diag = Ls(-1, -1) + Ls(-1, 1) + Ls(1, -1) + Ls(1, 1);
    const T ah = aH[i] + (T(4) * axis + diag - T(20) * Ls(0, 0)) / T(6);
    const T jx = aJx[i], jy = aJy[i], om = T(1) - C.omega;
#pragma unroll
    for (int l = 0; l < 9; ++l) {
        const T m = a_next[l * D.n + nb.at(aCy[l], aCx[l])];
        a[l * D.n + i] = ah + T(aCx[l]) * jx + T(aCy[l]) * jy + om * m;
    }
}

// dL/dh0 = sum_l a_l(0) dE_l(h0, 0)/dh0, which with a_l = aH + c_l . aJ (three
// fields, omega = 1) is aH; dL/dtheta = dL/dkappa sin(theta) c
template <typename T>
__global__ void k_adj_init(const T* __restrict__ h0, const T* __restrict__ a0, T* gh0, const T* __restrict__ gk,
                           const T* __restrict__ theta, T* gth, Dims D, Consts<T> C, T kc, T theta_u, bool three)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= D.n) return;
    if (gh0) {
        T s = a0[i];
        if (!three) {
            const T hh = h0[i];
            s *= T(1) - T(5) * C.g * hh / T(3);
#pragma unroll
            for (int l = 1; l < 9; ++l) s += a0[l * D.n + i] * C.g * hh * ((l & 1) ? T(1.0 / 3.0) : T(1.0 / 12.0));
        }
        gh0[i] = s;
    }
    if (gth) gth[i] = gk[i] * sin(theta ? theta[i] : theta_u) * kc;
}

// a(T) = dL/df(T): h = sum_l f_l, so aH = dL/dh, aJ = 0; dL/dkappa starts at 0
template <typename T>
__global__ void k_seed(const T* __restrict__ gh, T* a, T* gk, Dims D, bool three)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= D.n) return;
    const T v = gh[i];
    gk[i] = T(0);
    a[i] = v;
    if (three) {
        a[D.n + i] = T(0);
        a[2 * D.n + i] = T(0);
    } else {
#pragma unroll
        for (int l = 1; l < 9; ++l) a[l * D.n + i] = v;
    }
}

inline dim3 g2(const Dims& D) { return dim3((D.nx + 127) / 128, D.ny); }
inline int g1(const Dims& D) { return (int)((D.n + 255) / 256); }

template <typename T>
cudaError_t adjoint_t(tf_lbm_handle* H, const void* f, const void* an, void* a, void* gk, cudaStream_t st)
{
    Dims D{H->G.nx, H->G.ny, (long long)H->G.nx * H->G.ny};
    T* s = (T*)H->adj;
    T *h = s, *jx = s + D.n, *jy = s + 2 * D.n, *p = s + 3 * D.n, *aH = s + 4 * D.n, *aJx = s + 5 * D.n,
      *aJy = s + 6 * D.n, *agx = s + 7 * D.n, *agy = s + 8 * D.n, *alap = s + 9 * D.n;
    const Consts<T> C = make_consts<T>(H);
    const T* kap = (const T*)H->kappa;
    k_adj_moments<T><<<g2(D), 128, 0, st>>>((const T*)f, h, jx, jy, D);
    k_adj_pressure<T><<<g2(D), 128, 0, st>>>(h, kap, p, D, C);
    k_adj_collide<T><<<g2(D), 128, 0, st>>>(h, jx, jy, p, (const T*)an, aH, aJx, aJy, agx, agy, D, C);
    k_adj_pressure_t<T><<<g2(D), 128, 0, st>>>(agx, agy, h, kap, aH, alap, (T*)gk, D, C);
    k_adj_out<T><<<g2(D), 128, 0, st>>>(aH, alap, aJx, aJy, (const T*)an, (T*)a, D, C);
    return cudaGetLastError();
}

}  // namespace

cudaError_t adjoint_step_dispatch(tf_lbm_handle* H, const void* f, const void* an, void* a, void* gk,
                                  cudaStream_t st)
{
    if (!H->adj) {
        cudaError_t e = cudaMalloc(&H->adj, 10ull * H->G.nx * H->G.ny * H->esize);
        if (e != cudaSuccess) return e;
    }
    return H->dbl ? adjoint_t<double>(H, f, an, a, gk, st) : adjoint_t<float>(H, f, an, a, gk, st);
}

namespace {

template <typename S>
cudaError_t adjoint_tile_t(tf_lbm_handle* H, const void* mom, bool fresh, const void* an, void* a, void* gk, cudaStream_t st)
{
    const Consts<S> C = make_consts<S>(H);
    const S *m = (const S*)mom, *n = (const S*)an, *k = (const S*)H->kappa;
    switch (H->tape_tile ? H->tape_tile : adjoint_block_x(H->dbl, H->G.nx, H->G.ny, H->sms)) {
        case 64: return adjoint_tile_one<S, 16, 8>(m, fresh, n, (S*)a, (S*)gk, k, H->G, C, st);
        case 128: return adjoint_tile_one<S, 16, 16>(m, fresh, n, (S*)a, (S*)gk, k, H->G, C, st);
        default: return adjoint_tile_one<S, 32, 16>(m, fresh, n, (S*)a, (S*)gk, k, H->G, C, st);
    }
}

// One adjoint step from the record of its state.  fresh: the launch before this
// one may have written it.
cudaError_t adjoint_tile_step(tf_lbm_handle* H, const void* mom, bool fresh, const void* an, void* a,
                              void* gk, cudaStream_t st)
{
    return H->dbl ? adjoint_tile_t<double>(H, mom, fresh, an, a, gk, st)
                  : adjoint_tile_t<float>(H, mom, fresh, an, a, gk, st);
}

// omega == 1 in the compute type: three-field adjoint states
bool three_fields(const tf_lbm_handle* H)
{
    return H->dbl ? make_consts<double>(H).omega == 1.0 : make_consts<float>(H).omega == 1.0f;
}

}  // namespace

}  // namespace tflbm

// ---------------------------------------------------------------- the tape

// Largest set of step records a tape keeps in place of state copies and
// recomputation where these take less: 4 GiB, and 1/64 of the memory that is
// free when the tape is made.  Keeping all pays in time at any size (512^2: a step
// costs 5.2 us to recompute and its 3 MB 2 us to allocate and free), but a tape
// is not the only tenant: the caller's own allocations come after it, and many
// tapes may live at a time, each of which leaves 63/64 of what it found.
constexpr size_t kTapeBytes = (size_t)4 << 30;
constexpr size_t kTapeShare = 64;

struct tf_lbm_tape {
    tf_lbm_handle* H = nullptr;
    int64_t nsteps = 0;
    int every = 1;                 // records kept at a time: all steps, or one segment
    int nseg = 0;                  // segments of `every` steps (the last may be shorter)
    size_t state_bytes = 0;        // one raw population buffer
    size_t rec_bytes = 0;          // one record: h - href, j_x, j_y
    size_t a_bytes = 0;            // one adjoint state
    void* block = nullptr;         // one allocation for what follows
    void* ck = nullptr;            // states at 0, K, 2K, ... (nseg > 1), then two buffers to recompute in
    void* rec = nullptr;           // `every` records
    void* abuf = nullptr;          // 2 adjoint states
    void* gk = nullptr;            // dL/dkappa
    void* h0 = nullptr;            // copy of h0 (compute type)
    void* theta = nullptr;         // copy of theta or null (uniform)
    bool forwarded = false;
};

namespace {

int tape_fail(tf_lbm_tape* tp, int code, const char* msg) { return handle_fail(tp ? tp->H : nullptr, code, msg); }

#define TK(tp, call, what)                                                       \
    do {                                                                         \
        cudaError_t e_ = (call);                                                 \
        if (e_ != cudaSuccess) return handle_cuda_fail((tp)->H, e_, what);      \
    } while (0)

int64_t segment_steps(const tf_lbm_tape* tp, int c)
{
    return std::min<int64_t>(tp->every, tp->nsteps - (int64_t)c * tp->every);
}

// Write the records of a segment of len steps that starts at the copy c.
cudaError_t recompute(tf_lbm_tape* tp, int c, int64_t len, cudaStream_t st)
{
    char* ck = (char*)tp->ck;
    char* work = ck + tp->nseg * tp->state_bytes;
    const char* from = ck + c * tp->state_bytes;
    for (int64_t i = 0; i < len; ++i) {
        char* to = work + (i & 1) * tp->state_bytes;
        const cudaError_t e = launch_recorded_step(tp->H, from, to, (char*)tp->rec + i * tp->rec_bytes, st);
        if (e != cudaSuccess) return e;
        from = to;
    }
    return cudaSuccess;
}

}  // namespace

extern "C" {

int tf_lbm_adjoint_step(tf_lbm_handle* H, const void* f_t, const void* a_next, void* a_t, void* grad_kappa,
                        void* stream)
{
    if (!H) return handle_fail(nullptr, TF_LBM_ERR_ARG, "handle is NULL");
    if (!f_t || !a_next || !a_t || !grad_kappa)
        return handle_fail(H, TF_LBM_ERR_ARG, "f_t, a_next, a_t and grad_kappa must not be NULL");
    if (a_t == a_next) return handle_fail(H, TF_LBM_ERR_ARG, "a_t must not alias a_next");
    if (H->p.forcing != 0)
        return handle_fail(H, TF_LBM_ERR_UNSUPPORTED, "the adjoint differentiates Eq. (LBE) as printed (forcing = 0)");
    cudaError_t e = adjoint_step_dispatch(H, f_t, a_next, a_t, grad_kappa, (cudaStream_t)stream);
    if (e != cudaSuccess) return handle_cuda_fail(H, e, "adjoint kernels");
    return TF_LBM_OK;
}

int tf_lbm_tape_create(tf_lbm_handle* H, const void* h0, const void* theta, int64_t nsteps, int32_t every,
                       tf_lbm_tape** out)
{
    if (!H) return handle_fail(nullptr, TF_LBM_ERR_ARG, "handle is NULL");
    if (!out) return handle_fail(H, TF_LBM_ERR_ARG, "out must not be NULL");
    *out = nullptr;
    if (!h0) return handle_fail(H, TF_LBM_ERR_ARG, "h0 must not be NULL");
    if (nsteps < 1) return handle_fail(H, TF_LBM_ERR_ARG, "nsteps must be >= 1");
    if (H->p.forcing != 0)
        return handle_fail(H, TF_LBM_ERR_UNSUPPORTED, "the adjoint differentiates Eq. (LBE) as printed (forcing = 0)");
    const long long n = (long long)H->G.nx * H->G.ny;
    tf_lbm_tape* tp = new tf_lbm_tape();
    tp->H = H;
    tp->nsteps = nsteps;
    tp->state_bytes = (size_t)H->G.plane * (H->esize + 8 * H->msize);
    tp->rec_bytes = 3ull * n * H->esize;
    tp->a_bytes = (three_fields(H) ? 3ull : 9ull) * n * H->esize;
    cudaError_t e;
    auto bail = [&](cudaError_t err, const char* what) {
        int rc = handle_cuda_fail(H, err, what);
        tf_lbm_tape_destroy(tp);
        return rc;
    };
    // One allocation.  All records where they may be kept (every <= 0 leaves the
    // choice here; an explicit `every` asks for segments of that length), else
    // segments
    const size_t field = n * H->esize;
    const int64_t root = (int64_t)ceil(sqrt((double)nsteps));
    auto may_keep_all = [&]() {
        const size_t most = kTapeBytes / tp->rec_bytes;
        if (nsteps > INT32_MAX) return false;
        const size_t segments = tp->state_bytes * ((nsteps + root - 1) / root + 2) + tp->rec_bytes * root;
        if ((size_t)nsteps <= segments / tp->rec_bytes) return true;  // no more than segments would take
        size_t left = 0, total = 0;
        if ((size_t)nsteps > most || cudaMemGetInfo(&left, &total) != cudaSuccess) return false;
        return (size_t)nsteps <= left / kTapeShare / tp->rec_bytes;
    };
    auto allocate = [&](int64_t kept) {
        tp->every = (int)kept;
        tp->nseg = (int)((nsteps + kept - 1) / kept);
        Carver cut;
        const size_t at_a = cut.take(2 * tp->a_bytes), at_gk = cut.take(field), at_h0 = cut.take(field);
        const size_t at_theta = cut.take(theta ? field : 0);
        const size_t at_ck = cut.take(tp->nseg > 1 ? tp->state_bytes * (tp->nseg + 2) : 0);
        const size_t at_rec = cut.take(tp->rec_bytes * kept);
        const cudaError_t err = cudaMalloc(&tp->block, cut.total);
        if (err != cudaSuccess) {
            tp->block = nullptr;
            return err;
        }
        char* block = (char*)tp->block;
        tp->abuf = block + at_a;
        tp->gk = block + at_gk;
        tp->h0 = block + at_h0;
        tp->theta = theta ? block + at_theta : nullptr;
        tp->ck = block + at_ck;
        tp->rec = block + at_rec;
        return cudaSuccess;
    };
    if (every <= 0 && may_keep_all() && allocate(nsteps) != cudaSuccess) cudaGetLastError();
    if (!tp->block) {
        if (every <= 0) every = (int32_t)root;
        if ((e = allocate(std::min<int64_t>(every, nsteps))) != cudaSuccess) return bail(e, "cudaMalloc tape");
    }
    if ((e = cudaMemcpy(tp->h0, h0, field, cudaMemcpyDeviceToDevice)) != cudaSuccess) return bail(e, "copy h0");
    if (theta && (e = cudaMemcpy(tp->theta, theta, field, cudaMemcpyDeviceToDevice)) != cudaSuccess)
        return bail(e, "copy theta");
    *out = tp;
    return TF_LBM_OK;
}

int tf_lbm_tape_forward(tf_lbm_tape* tp, void* stream)
{
    if (!tp) return handle_fail(nullptr, TF_LBM_ERR_ARG, "tape is NULL");
    tf_lbm_handle* H = tp->H;
    cudaStream_t st = (cudaStream_t)stream;
    for (int c = 0; c < tp->nseg; ++c) {
        if (tp->nseg > 1)
            TK(tp, cudaMemcpyAsync((char*)tp->ck + c * tp->state_bytes, H->buf[H->cur], tp->state_bytes,
                                   cudaMemcpyDeviceToDevice, st), "checkpoint copy");
        const int64_t len = segment_steps(tp, c);
        for (int64_t i = 0; i < len; ++i) {
            TK(tp, launch_recorded_step(H, H->buf[H->cur], H->buf[H->cur ^ 1], (char*)tp->rec + i * tp->rec_bytes, st),
               "step kernel");
            H->cur ^= 1;
            ++H->time;
        }
    }
    tp->forwarded = true;
    return TF_LBM_OK;
}

int tf_lbm_tape_backward(tf_lbm_tape* tp, const void* grad_h, void* grad_theta, void* grad_h0, void* stream)
{
    if (!tp) return handle_fail(nullptr, TF_LBM_ERR_ARG, "tape is NULL");
    tf_lbm_handle* H = tp->H;
    if (!tp->forwarded) return tape_fail(tp, TF_LBM_ERR_ARG, "tf_lbm_tape_forward must run first");
    if (!grad_h) return tape_fail(tp, TF_LBM_ERR_ARG, "grad_h must not be NULL");
    cudaStream_t st = (cudaStream_t)stream;
    const long long n = (long long)H->G.nx * H->G.ny;
    char* ab = (char*)tp->abuf;
    const bool three = three_fields(H);
    Dims D{H->G.nx, H->G.ny, n};
    int cur = 0;  // adjoint state in ab + cur * a_bytes
    if (H->dbl) k_seed<double><<<g1(D), 256, 0, st>>>((const double*)grad_h, (double*)ab, (double*)tp->gk, D, three);
    else k_seed<float><<<g1(D), 256, 0, st>>>((const float*)grad_h, (float*)ab, (float*)tp->gk, D, three);
    TK(tp, cudaGetLastError(), "seed kernel");
    for (int c = tp->nseg - 1; c >= 0; --c) {
        const int64_t len = segment_steps(tp, c);
        if (tp->nseg > 1) TK(tp, recompute(tp, c, len, st), "recompute");
        for (int64_t i = len - 1; i >= 0; --i) {
            TK(tp, adjoint_tile_step(H, (char*)tp->rec + i * tp->rec_bytes, i == len - 1, ab + cur * tp->a_bytes,
                                     ab + (cur ^ 1) * tp->a_bytes, tp->gk, st), "adjoint step");
            cur ^= 1;
        }
    }
    if (grad_h0 || grad_theta) {
        const double kc = (double)(H->p.n_exp - 1) * (H->p.m_exp - 1) / ((double)(H->p.n_exp - H->p.m_exp) * H->p.hstar);
        const void* a0 = ab + cur * tp->a_bytes;
        if (H->dbl)
            k_adj_init<double><<<g1(D), 256, 0, st>>>((const double*)tp->h0, (const double*)a0, (double*)grad_h0,
                                                      (const double*)tp->gk, (const double*)tp->theta,
                                                      (double*)grad_theta, D, make_consts<double>(H), kc,
                                                      H->p.theta_uniform, three);
        else
            k_adj_init<float><<<g1(D), 256, 0, st>>>((const float*)tp->h0, (const float*)a0, (float*)grad_h0,
                                                     (const float*)tp->gk, (const float*)tp->theta,
                                                     (float*)grad_theta, D, make_consts<float>(H), (float)kc,
                                                     (float)H->p.theta_uniform, three);
        TK(tp, cudaGetLastError(), "init adjoint kernel");
    }
    return TF_LBM_OK;
}

void tf_lbm_tape_destroy(tf_lbm_tape* tp)
{
    if (!tp) return;
    cudaDeviceSynchronize();
    if (tp->block) cudaFree(tp->block);
    delete tp;
}

}  // extern "C"
