// C-ABI of the thin-film D2Q9 lattice Boltzmann library (include/tflbm.h).
// Owns the population ping-pong buffers, the kappa field and the reduction
// scratch; launches the fused step kernel once per time step, optionally
// replaying a captured CUDA graph of an even number of steps.
#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <string>

#include "../../include/tflbm.h"
#include "tflbm_handle.h"

using namespace tflbm;

namespace tflbm {
int sm_count()
{
    int sms = 152, dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

static int rows_covered(int bx, int ny) { return (ny + tile_of(bx).ty - 1) / tile_of(bx).ty * tile_of(bx).ty; }
static long long tiles_of(int bx, int nx, int ny)
{
    const TileShape t = tile_of(bx);
    return (long long)((nx + t.tx - 1) / t.tx) * ((ny + t.ty - 1) / t.ty);
}

// The FP32 shape with the least work on the busiest SM, counting a node's pull
// as 0.45 of its cost and its pressure as 0.2 (the halos repeat those) and 60
// nodes' worth of fixed latency a tile.  Measured, one box, us a step with block_x
// 64 / 128 / 256: 64^2 2.34 / 2.40 / 2.46, 128^2 2.53 / 2.50 / 2.59, 200 x 150 3.16 / 2.90 /
// 2.94, 384^2 3.94 / 3.77 / 3.51, 512^2 6.92 / 6.62 / 4.53, 1024^2 20.7 / 20.2 / 15.1 (where
// 32 x 16 tiles run four an SM, see tile_one).
static int tile_block_f32(int nx, int ny, int sms)
{
    int best = 64;
    double least = 0;
    for (int bx : {64, 128, 256}) {
        const TileShape t = tile_of(bx);
        const double work = 60 + 0.35 * t.tx * t.ty + 0.45 * (t.tx + 4) * (t.ty + 4) + 0.2 * (t.tx + 2) * (t.ty + 2);
        const double cost = (double)((tiles_of(bx, nx, ny) + sms - 1) / sms) * work;
        if (bx == 64 || cost < least) {
            best = bx;
            least = cost;
        }
    }
    return best;
}

// The tile kernel's block_x for a lattice (tile_of).  FP32: as above, but 16 x 8
// tiles on long lattices of a few rows, of which 16-row tiles would cover over 1.2
// times as many (block_x 64 / 256: 60000 x 20 28.3 / 30.9, 20000 x 24 10.9 / 11.2, 30000
// x 33, 1.2 times, 22.9 / 21.8).  FP64 is bound by its arithmetic units: the least
// tiles times the cost of one, of which the halos are a smaller part the larger it
// is, but the small ones, which spread best over the SMs, up to six an SM.  Us a
// step with block_x 64 / 128 / 256: 100^2 8.2 / 12.8 / 22.2, 250 x 190 18.3 / 23.0 /
// 22.4, 400 x 300 40.1 / 43.9 / 43.7, 512^2 78 / 76 / 85, 2048^2 1175 / 1135 / 1179, 60000 x
// 20 409 / 525 / 549; omega = 1: 512^2 - / 70 / 77, 3000 x 500 396 / 389 / 378.
int tile_block_x(int store, int nx, int ny, int sms, bool omega1)
{
    if (store != kStoreF64) {
        if ((long long)nx * rows_covered(256, ny) >= 1LL << 19 && 5 * rows_covered(256, ny) > 6 * rows_covered(64, ny))
            return 64;
        return tile_block_f32(nx, ny, sms);
    }
    const double small = (double)tiles_of(64, nx, ny), mid = 1.93 * tiles_of(128, nx, ny),
                 large = (omega1 ? 3.76 : 4.0) * tiles_of(256, nx, ny);
    if (small <= 6.0 * sms || (small <= mid && small <= large)) return 64;
    return mid <= large || tiles_of(256, nx, ny) < 7LL * sms ? 128 : 256;
}
// The adjoint's tiles, whose halos are one node deeper.
int adjoint_block_x(bool dbl, int nx, int ny, int sms)
{
    if (!dbl) return tile_block_f32(nx, ny, sms);
    if (5 * rows_covered(256, ny) > 6 * rows_covered(64, ny)) return 64;
    return tiles_of(64, nx, ny) <= sms ? 64 : (tiles_of(256, nx, ny) >= 7LL * sms ? 256 : 128);
}
}  // namespace tflbm

namespace {

thread_local std::string g_init_err;

int fail(tf_lbm_handle* H, int code, const std::string& msg)
{
    if (H) H->err = msg;
    else g_init_err = msg;
    return code;
}

int cuda_fail(tf_lbm_handle* H, cudaError_t e, const char* what)
{
    std::string m = std::string(what) + ": " + cudaGetErrorName(e) + " (" + cudaGetErrorString(e) + ")";
    return fail(H, e == cudaErrorMemoryAllocation ? TF_LBM_ERR_NOMEM : TF_LBM_ERR_CUDA, m);
}

#define CK(H, call, what)                                  \
    do {                                                   \
        cudaError_t e_ = (call);                           \
        if (e_ != cudaSuccess) return cuda_fail(H, e_, what); \
    } while (0)

// Device pointers only: host memory handed to a kernel would fault or read
// the wrong memory.
int check_dev_ptr(tf_lbm_handle* H, const void* ptr, const char* name, bool allow_null)
{
    if (!ptr) {
        if (allow_null) return TF_LBM_OK;
        return fail(H, TF_LBM_ERR_ARG, std::string(name) + " must not be NULL");
    }
    cudaPointerAttributes a;
    cudaError_t e = cudaPointerGetAttributes(&a, ptr);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(H, TF_LBM_ERR_ARG, std::string(name) + " is not a CUDA pointer");
    }
    if (a.type != cudaMemoryTypeDevice && a.type != cudaMemoryTypeManaged)
        return fail(H, TF_LBM_ERR_ARG, std::string(name) + " must be device or managed memory");
    int dev = 0;
    cudaGetDevice(&dev);
    if (a.type == cudaMemoryTypeDevice && a.device != dev)
        return fail(H, TF_LBM_ERR_ARG, std::string(name) + " lives on another device");
    return TF_LBM_OK;
}

void drop_graphs(tf_lbm_handle* H)
{
    for (auto& e : H->exec)
        if (e) {
            cudaGraphExecDestroy(e);
            e = nullptr;
        }
}

int validate(const tf_lbm_params* p)
{
    char buf[256];
    auto bad = [&](const char* m) {
        snprintf(buf, sizeof buf, "invalid parameter: %s", m);
        g_init_err = buf;
        return TF_LBM_ERR_ARG;
    };
    if (!p) return bad("params is NULL");
    if (p->nx < 1 || p->ny < 1) return bad("nx and ny must be >= 1");
    if (p->ny > 65535) return bad("ny must be <= 65535");
    if ((long long)p->nx * p->ny > (1LL << 31)) return bad("nx * ny must be <= 2^31");
    if (p->dtype != TF_LBM_F32 && p->dtype != TF_LBM_F64 && p->dtype != TF_LBM_F16 && p->dtype != TF_LBM_BF16)
        return bad("dtype must be TF_LBM_F32, TF_LBM_F64, TF_LBM_F16 or TF_LBM_BF16");
    if (!(p->tau > 0.5)) return bad("tau must be > 1/2");
    if (!(p->hstar > 0.0)) return bad("hstar must be > 0");
    if (!(p->delta >= 0.0)) return bad("delta must be >= 0");
    if (p->n_exp < 1 || p->m_exp < 1 || p->n_exp > 64 || p->m_exp > 64) return bad("n_exp and m_exp must be in [1, 64]");
    if (p->n_exp == p->m_exp) return bad("n_exp must differ from m_exp");
    if (p->pi_sign != 1 && p->pi_sign != -1) return bad("pi_sign must be +1 or -1");
    if (p->forcing != 0 && p->forcing != 1) return bad("forcing must be 0 or 1");
    if (!isfinite(p->gamma) || !isfinite(p->g) || !isfinite(p->gx_body) || !isfinite(p->gy_body) ||
        !isfinite(p->theta_uniform) || !isfinite(p->tau))
        return bad("non-finite parameter");
    return TF_LBM_OK;
}

// Whether a run's steps go one by one to the two-column march, which has the
// same bits: short runs of the four-column march in the ragged layout, whose first
// and last step, from and to populations, cost more than the steps between them
// save (us a step in runs of two, two-column / four-column: 362 x 11602 58.1 / 76.0, 602
// x 6976 55.5 / 68.9, 1030 x 4077 55.9 / 61.3, 2046^2 52.7 / 54.3; in runs of eight the
// two are even).
bool one_by_one(const tf_lbm_handle* H, int64_t steps)
{
    return H->shape.wide && H->desc.store == kStoreF32 && H->G.nx % 4 == 2 && steps < 8;
}

int store_of(int dtype)
{
    switch (dtype) {
        case TF_LBM_F64: return kStoreF64;
        case TF_LBM_F16: return kStoreF16;
        case TF_LBM_BF16: return kStoreBF16;
        default: return kStoreF32;
    }
}

// The tile kernel runs where its rows cover at most this many nodes in place of:
// the four-column march (nx a multiple of 4; ragged), the two-column march of
// narrow 16-bit lattices, the other marches (tau != 1, forcing, narrow ragged
// lattices).  FP64, and 16-bit storage where the one-column march is what is left,
// run tiles at any size.  Above the limits the marches win: they pull a node 1.25
// times, not 1.4, and load ahead.  Us a step, tile against march: FP32 four-column
// 900^2 12.7 / 13.2, 1028^2 17.1 / 17.3, 1064^2 18.5 / 17.3, 1448^2 36.9 / 22.3; ragged 1030 x 1067 17.9 /
// 21.4, 1205 x 1078 22.8 / 22.0, 1030 x 1262 23.1 / 22.2; FP16 1028^2 16.8 / 17.3, 1100^2
// 18.3 / 17.6, 1448^2 31.8 / 21.6; against the one-column march at tau = 0.8: FP32 1228^2
// 27.6 / 39.0, 1448^2 37.3 / 39.7, 1700^2 49.8 / 47.3, 2048^2 69 / 64, FP16 1448^2 32.7 /
// 45.0, 2048^2 59.9 / 71.7; FP64 2048^2 1135 / 1372.
constexpr long long kTileQuad = 17LL << 16, kTileRagged = 5LL << 18, kTileMarch = 3LL << 19;

// Long lattices of a few rows, of which tiles cover too many: they cost more than
// the latency of a march's few rows (us a step, tile of the best shape against
// march; nodes covered, thousands, of those in the lattice): FP64 65000 x 17 408 /
// 338 (1560 of 1105), 40000 x 9 165 / 141 (640 of 360), 20000 x 9 88 / 118 (320 of
// 180), 30000 x 3 73 / 46 (240 of 90), 60000 x 20 378 / 394 (1440 of 1200); FP32 100000
// x 3 15.0 / 11.5 (800 of 300), 30000 x 3 6.7 / 6.2 (240 of 90), 40000 x 9 10.7 / 14.7,
// 65000 x 17 31 / 29, 30000 x 33 21.9 / 28.8 (1440 of 990), 60000 x 20 28 / 36 in long
// runs, 30.6 / 25.8 in runs of two.
bool tiles_wasted(int store, long long covered, long long nodes)
{
    if (3 * covered <= 4 * nodes) return false;
    if (store == kStoreF64) return covered - nodes > 9LL << 14;
    return covered > 1500000 || (covered > 2 * nodes && covered - nodes > 1LL << 17);
}

// Whether the four-column march beats the others on a lattice that it takes.
// Ragged: its strips at either end of a row, which load and store by nodes, have
// to be few beside the others (us a step in runs of 20, two-column / four-column:
// 122 x 24590 44.9 / 57.8, 126 x 17460 43.3 / 45.0, 242 x 17355 58.0 / 61.5, 242 x 9090 39.9 /
// 36.5, 362 x 11602 56.5 / 57.5, 362 x 6077 39.7 / 34.3, 482 x 8713 56.0 / 54.5, 1030 x 4077
// 54.6 / 48.0; one-column, nx odd: 483 x 4554 36.4 / 32.5, 2047 x 2049 60 / 45, 243 x 9053
// 38.7 / 36.3, but 40.6 / 47.8 in runs of two).  A run of one step, which tiles take
// where nx is odd, costs more than the one-column march there: 2047 x 2049 74 / 65.
bool wide_wins(int store, const Geom& G)
{
    WideCover cover;
    cover.add(G.nx, G.ny);
    if (G.nx % 4 == 0) return cover.pays(store);
    const int strips = wide_strips(G.nx);
    return strips >= 5 || (strips >= 3 && G.nx % 2 == 0 && (long long)G.nx * G.ny <= 3LL << 20);
}

// A march filled with balanced bands: as many as fill the resident slots once
// (all bands do the same work, so a partial second wave would idle most SMs),
// but none shorter than 16 rows: each band spends 5 warm-up rows.
void fill_bands(Shape& s, int store, const Geom& G, bool om1, bool kfield, int sms)
{
    const int strips = (G.nx + s.block_x - 5) / (s.block_x - 4);  // CTAs overlap by 4 columns
    int occ = step_blocks_per_sm(store, s.pipeline, s.block_x, om1, kfield);
    if (occ < 1) occ = 4;
    int bands = occ * sms / strips;
    if (bands > G.ny / 16) bands = G.ny / 16;
    if (bands < 1) bands = 1;
    if (bands > 65535) bands = 65535;
    s.bands = bands;
    s.rows = (G.ny + bands - 1) / bands;
}

// Default launch shape: tiles on lattices that L2 holds, the four-column march
// on larger ones at tau = 1, by the rules above.  The other fields describe the
// march that is left: the two-column kernel at tau = 1 where it applies
// (CTAs 64 columns wide for 16-bit storage, 128 for FP32), else the one-column kernel
// with CTAs 128 columns wide (64 on lattices narrower than 1024).
Shape default_shape(const tf_lbm_params& p, const Geom& G, bool kfield)
{
    Shape s;
    // two columns per thread at tau = 1 where pairs fit (nx even): it issues
    // fewer instructions per node than the one-column kernel, which is issue
    // bound; 16-bit storage uses it at 64 columns per CTA (one warp), FP32 at
    // 128.  At tau != 1 the one-column kernel is faster in every storage type
    // (the two-column kernel's pulled-population ring costs resident warps)
    const int store = store_of(p.dtype), sms = sm_count();
    const bool om1 = p.tau == 1.0;
    const bool quad = G.nx % 4 == 0;
    const bool wide = om1 && p.forcing == 0 && wide_applies(store, G, quad) && wide_wins(store, G);
    const bool pair = pair_pipeline_ok(G.nx, store) && om1;
    const bool narrow = store == kStoreF16 || store == kStoreBF16;
    const int bx = tile_block_x(store, G.nx, G.ny, sms, om1);
    const long long covered = (long long)G.nx * rows_covered(bx, G.ny);
    const long long limit = wide ? (quad ? kTileQuad : kTileRagged) : (narrow && pair && quad ? kTileQuad : kTileMarch);
    if ((store == kStoreF64 || (narrow && !wide && !pair) || covered <= limit) &&
        !tiles_wasted(store, covered, (long long)G.nx * G.ny))
        s.tile = bx;
    else if (wide)
        s.wide = wide_bands(G, wide_slots(store, quad, sms));
    s.block_x = pair ? (narrow ? 64 : 128) : (G.nx >= 1024 ? 128 : 64);
    // otherwise per-thread loads: measured faster than the bulk-copy pipeline
    // on GB300 once loads are prefetched a row ahead
    s.pipeline = pair ? kPipePair : kPipeLdg;
    fill_bands(s, store, G, om1, kfield, sms);
    return s;
}

}  // namespace

namespace tflbm {
// Message for tf_lbm_last_error(NULL) from entry points without a handle.
void set_thread_error(const std::string& msg) { g_init_err = msg; }

int handle_fail(tf_lbm_handle* H, int code, const std::string& msg) { return fail(H, code, msg); }
int handle_check_dev_ptr(tf_lbm_handle* H, const void* ptr, const char* name, bool allow_null)
{
    return check_dev_ptr(H, ptr, name, allow_null);
}
void handle_drop_graphs(tf_lbm_handle* H) { drop_graphs(H); }
int handle_cuda_fail(tf_lbm_handle* H, cudaError_t e, const char* what) { return cuda_fail(H, e, what); }

template <typename T>
Consts<T> make_consts(const tf_lbm_handle* H)
{
    Consts<T> C;
    C.gamma = T(H->p.gamma);
    C.g = T(H->p.g);
    C.delta = T(H->p.delta);
    C.hstar = T(H->p.hstar);
    C.nu6 = T(6.0 * (H->p.tau - 0.5) / 3.0);
    C.omega = T(1.0 / H->p.tau);
    C.gx = T(H->p.gx_body);
    C.gy = T(H->p.gy_body);
    C.kappa_u = T(H->kappa_u);
    C.pi_sgn = T(H->p.pi_sign);
    C.href = T(H->href);
    C.mscale = T(H->desc.mscale);
    C.minv = T(H->desc.minv);
    C.r_axis = T(H->desc.r_axis);
    C.r_diag = T(H->desc.r_diag);
    C.nr_axis = T(-H->desc.r_axis * H->desc.mscale);
    C.nr_diag = T(-H->desc.r_diag * H->desc.mscale);
    C.r_sum = T(4.0 * (H->desc.r_axis + H->desc.r_diag));
    C.n_exp = H->p.n_exp;
    C.m_exp = H->p.m_exp;
    C.status = H->status;
    C.wait_limit = H->wait_limit;
    C.forcing = H->p.forcing;
    C.flip = 0;
    return C;
}

cudaError_t launch_one_step(tf_lbm_handle* H, int from, cudaStream_t st, bool first, bool last)
{
    Consts<float> c32 = make_consts<float>(H);
    Consts<double> c64 = make_consts<double>(H);
    c32.flip = c64.flip = from & 1;
    if (H->shape.wide) {
        const bool f32 = H->desc.store == kStoreF32;
        if (!(f32 && first && last))
            return launch_wide(H->desc.store, f32 && !first, f32 && !last, H->buf[from], H->buf[from ^ 1], H->kappa, H->G,
                               c32, H->shape.wide, st);
        // A run of one FP32 step has no moments to keep: the two-column march
        // (2048^2: 53 against 56 us), or tiles where nx is odd; same bits,
        // whatever march the shape was put in place of.
        if (!pair_pipeline_ok(H->G.nx, kStoreF32))
            return launch_tile(H->desc.store, 256, H->buf[from], H->buf[from ^ 1], H->kappa, nullptr, H->G, &c32, &c64, st);
        return launch_step(H->desc.store, H->buf[from], H->buf[from ^ 1], H->kappa, H->G, &c32, &c64, H->one, st);
    }
    return launch_step(H->desc.store, H->buf[from], H->buf[from ^ 1], H->kappa, H->G, &c32, &c64,
                       H->shape, st);
}

cudaError_t launch_recorded_step(tf_lbm_handle* H, const void* fin, void* fout, void* mom, cudaStream_t st)
{
    const Consts<float> c32 = make_consts<float>(H);
    const Consts<double> c64 = make_consts<double>(H);
    const bool om1 = H->dbl ? c64.omega == 1.0 : c32.omega == 1.0f;
    const int bx = H->tape_tile ? H->tape_tile : tile_block_x(H->desc.store, H->G.nx, H->G.ny, H->sms, om1);
    return launch_tile(H->desc.store, bx, fin, fout, H->kappa, mom, H->G, &c32, &c64, st);
}

template Consts<float> make_consts<float>(const tf_lbm_handle*);
template Consts<double> make_consts<double>(const tf_lbm_handle*);
}  // namespace tflbm

static_assert(kStatusTimeout == TF_LBM_STATUS_TIMEOUT, "status bits out of sync");

extern "C" {

int32_t tf_lbm_version(void) { return 200; }

const char* tf_lbm_last_error(const tf_lbm_handle* H)
{
    return H ? H->err.c_str() : g_init_err.c_str();
}

int tf_lbm_init(tf_lbm_handle** out, const tf_lbm_params* params, const void* h0,
                const void* theta, void* stream)
{
    g_init_err.clear();
    if (!out) return fail(nullptr, TF_LBM_ERR_ARG, "out must not be NULL");
    *out = nullptr;
    int rc = validate(params);
    if (rc) return rc;
    if ((rc = check_dev_ptr(nullptr, h0, "h0", false))) return rc;
    if ((rc = check_dev_ptr(nullptr, theta, "theta", true))) return rc;

    tf_lbm_handle* H = new tf_lbm_handle();
    H->p = *params;
    cudaStream_t st = (cudaStream_t)stream;
    cudaGetDevice(&H->device);
    H->desc.store = store_of(params->dtype);
    H->dbl = params->dtype == TF_LBM_F64;
    H->esize = H->dbl ? 8 : 4;
    H->msize = (params->dtype == TF_LBM_F16 || params->dtype == TF_LBM_BF16) ? 2 : H->esize;
    const int align = 128 / (int)H->msize;  // rows of every plane start on 128-byte boundaries
    H->G.nx = params->nx;
    H->G.ny = params->ny;
    H->G.pitch = (params->nx + align - 1) / align * align;
    H->G.plane = (long long)params->ny * H->G.pitch;
    if (9LL * H->G.plane >= (1LL << 31)) {  // the step kernel uses 32-bit element offsets
        delete H;
        return fail(nullptr, TF_LBM_ERR_UNSUPPORTED,
                    "lattice too large: 9 * ny * pitch must stay below 2^31 elements");
    }
    H->sms = sm_count();
    H->shape = H->def = H->own = default_shape(*params, H->G, theta != nullptr);
    if (H->desc.store == kStoreF32 && pair_pipeline_ok(H->G.nx, kStoreF32))
        fill_bands(H->one, kStoreF32, H->G, true, theta != nullptr, H->sms);
    H->graph_chunk = ((long long)params->nx * params->ny <= (1LL << 20)) ? 64 : 0;

    auto bail = [&](int code) {
        g_init_err = H->err;
        tf_lbm_destroy(H);
        return code;
    };
    // one allocation (35 to 80 us each to make and to free, of which a gradient's
    // handle and tape took sixteen): populations and flag, which start at zero,
    // then kappa and the reduction scratch
    const size_t bytes = (size_t)H->G.plane * (H->esize + 8 * H->msize);
    const long long n = (long long)params->nx * params->ny;
    H->nmass = mass_blocks(H->G);
    if (H->nmass < kSumBlocks) H->nmass = kSumBlocks;
    Carver cut;
    const size_t at0 = cut.take(bytes), at1 = cut.take(bytes), at_flag = cut.take(2 * sizeof(int)), zeros = cut.total;
    const size_t at_kappa = cut.take(theta ? n * H->esize : 0);
    const size_t at_partials = cut.take(sizeof(double) * 2 * H->nmass + sizeof(double));
    cudaError_t e;
    if ((e = cudaMalloc(&H->block, cut.total)) != cudaSuccess) return bail(cuda_fail(H, e, "cudaMalloc populations"));
    char* block = (char*)H->block;
    H->buf[0] = block + at0;
    H->buf[1] = block + at1;
    H->flag = (int*)(block + at_flag);
    H->status = H->flag + 1;
    H->partials = (double*)(block + at_partials);
    H->result = H->partials + 2 * H->nmass;
    if ((e = cudaMemsetAsync(H->block, 0, zeros, st)) != cudaSuccess) return bail(cuda_fail(H, e, "cudaMemsetAsync"));

    const double kscale = (double)(params->n_exp - 1) * (params->m_exp - 1) /
                          ((double)(params->n_exp - params->m_exp) * params->hstar);
    if (theta) {
        H->kappa = block + at_kappa;
        e = aux_kappa(H->dbl, H->kappa, theta, params->nx, params->ny, params->n_exp, params->m_exp,
                      params->hstar, st);
        if (e != cudaSuccess) return bail(cuda_fail(H, e, "kappa kernel"));
    } else {
        H->kappa_u = (1.0 - cos(params->theta_uniform)) * kscale;
    }
    // Reference height: the smallest h0, rounded to the storage type.  Plane
    // 0 stores f_0 - href, so FP32 resolves h - href to 2^-24 of |h - href|:
    // the thin parts of a film (precursor, contact lines), where the
    // disjoining pressure is stiffest and rounding differences grow fastest,
    // get the finest resolution, while thick parts keep 2^-24 relative.
    e = aux_min(H->dbl, h0, n, H->partials, H->nmass, H->result, st);
    if (e != cudaSuccess) return bail(cuda_fail(H, e, "min kernel"));
    double hmin = 0.0;
    if ((e = cudaMemcpyAsync(&hmin, H->result, sizeof(double), cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
        (e = cudaStreamSynchronize(st)) != cudaSuccess)
        return bail(cuda_fail(H, e, "reading the smallest height"));
    H->href = H->dbl ? hmin : (double)(float)hmin;
    if (!isfinite(H->href)) H->href = 0.0;  // a non-finite h0 is reported by tf_lbm_check
    // 16-bit storage of the moving populations: deviations from the rest
    // equilibrium at href, scaled by 2^10 in FP16 (keeps small deviations out
    // of the subnormal range; |f_l| up to 64 stays finite), unscaled in BF16.
    H->desc.href = H->href;
    H->desc.mscale = params->dtype == TF_LBM_F16 ? 1024.0 : 1.0;
    H->desc.minv = 1.0 / H->desc.mscale;
    if (H->msize == 2) {
        H->desc.r_axis = (double)(float)(params->g * H->href * H->href / 6.0);
        H->desc.r_diag = (double)(float)(params->g * H->href * H->href / 24.0);
    }
    e = aux_init(H->desc, H->buf[0], h0, H->G, params->g, st);
    if (e != cudaSuccess) return bail(cuda_fail(H, e, "init kernel"));
    H->cur = 0;
    *out = H;
    return TF_LBM_OK;
}

int tf_lbm_step(tf_lbm_handle* H, int64_t nsteps, void* stream)
{
    if (!H) return fail(nullptr, TF_LBM_ERR_ARG, "handle is NULL");
    if (nsteps < 0) return fail(H, TF_LBM_ERR_ARG, "nsteps must be >= 0");
    cudaStream_t st = (cudaStream_t)stream;
    const int chunk = H->graph_chunk;
    while (nsteps > 0) {
        if (chunk > 0 && nsteps >= chunk) {
            cudaGraphExec_t& ex = H->exec[H->cur];
            if (!ex) {
                if (!H->cap) CK(H, cudaStreamCreateWithFlags(&H->cap, cudaStreamNonBlocking), "cudaStreamCreate");
                CK(H, cudaStreamBeginCapture(H->cap, cudaStreamCaptureModeThreadLocal), "cudaStreamBeginCapture");
                cudaError_t le = cudaSuccess;
                const bool alone = one_by_one(H, chunk);
                for (int i = 0; i < chunk && le == cudaSuccess; ++i)
                    le = launch_one_step(H, H->cur ^ (i & 1), H->cap, alone || i == 0, alone || i == chunk - 1);
                cudaGraph_t g = nullptr;
                cudaError_t ce = cudaStreamEndCapture(H->cap, &g);
                if (le != cudaSuccess) { if (g) cudaGraphDestroy(g); return cuda_fail(H, le, "step kernel (capture)"); }
                if (ce != cudaSuccess) return cuda_fail(H, ce, "cudaStreamEndCapture");
                cudaError_t ie = cudaGraphInstantiate(&ex, g, 0);
                cudaGraphDestroy(g);
                if (ie != cudaSuccess) { ex = nullptr; return cuda_fail(H, ie, "cudaGraphInstantiate"); }
            }
            CK(H, cudaGraphLaunch(ex, st), "cudaGraphLaunch");
            nsteps -= chunk;
            H->time += chunk;
        } else {
            // one run of all the steps that no graph takes
            const bool alone = one_by_one(H, nsteps);
            for (const int64_t n = nsteps; nsteps > 0; --nsteps) {
                CK(H, launch_one_step(H, H->cur, st, alone || nsteps == n, alone || nsteps == 1), "step kernel");
                H->cur ^= 1;
                ++H->time;
            }
        }
    }
    return TF_LBM_OK;
}

int tf_lbm_moments(tf_lbm_handle* H, void* h, void* ux, void* uy, void* stream)
{
    if (!H) return fail(nullptr, TF_LBM_ERR_ARG, "handle is NULL");
    int rc;
    if ((rc = check_dev_ptr(H, h, "h", true)) || (rc = check_dev_ptr(H, ux, "ux", true)) ||
        (rc = check_dev_ptr(H, uy, "uy", true)))
        return rc;
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e = aux_moments(H->desc, H->buf[H->cur], h, ux, uy, H->G, st);
    CK(H, e, "moments kernel");
    return TF_LBM_OK;
}

int tf_lbm_pressure_force(tf_lbm_handle* H, void* p, void* fx, void* fy, void* stream)
{
    if (!H) return fail(nullptr, TF_LBM_ERR_ARG, "handle is NULL");
    int rc;
    if ((rc = check_dev_ptr(H, p, "p", true)) || (rc = check_dev_ptr(H, fx, "fx", true)) ||
        (rc = check_dev_ptr(H, fy, "fy", true)))
        return rc;
    cudaStream_t st = (cudaStream_t)stream;
    const Consts<float> c32 = make_consts<float>(H);
    const Consts<double> c64 = make_consts<double>(H);
    cudaError_t e = aux_pressure_force(H->desc, H->buf[H->cur], H->kappa, p, fx, fy, H->G, &c32, &c64, st);
    CK(H, e, "pressure/force kernel");
    return TF_LBM_OK;
}

int tf_lbm_mass(tf_lbm_handle* H, double* mass_host, void* stream)
{
    if (!H) return fail(nullptr, TF_LBM_ERR_ARG, "handle is NULL");
    if (!mass_host) return fail(H, TF_LBM_ERR_ARG, "mass_host must not be NULL");
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e = aux_mass(H->desc, H->buf[H->cur], H->G, H->partials, H->nmass, H->result, st);
    CK(H, e, "mass kernels");
    CK(H, cudaMemcpyAsync(mass_host, H->result, sizeof(double), cudaMemcpyDeviceToHost, st), "cudaMemcpyAsync");
    CK(H, cudaStreamSynchronize(st), "cudaStreamSynchronize");
    // plane 0 stores f_0 - href: add href back once per node
    *mass_host += H->href * (double)H->G.nx * (double)H->G.ny;
    return TF_LBM_OK;
}

int tf_lbm_check(tf_lbm_handle* H, int32_t* status_host, void* stream)
{
    if (!H) return fail(nullptr, TF_LBM_ERR_ARG, "handle is NULL");
    if (!status_host) return fail(H, TF_LBM_ERR_ARG, "status_host must not be NULL");
    cudaStream_t st = (cudaStream_t)stream;
    CK(H, cudaMemsetAsync(H->flag, 0, sizeof(int), st), "cudaMemsetAsync");
    cudaError_t e = aux_check(H->desc, H->buf[H->cur], H->G, H->flag, st);
    CK(H, e, "check kernel");
    int v[2] = {0, 0};
    CK(H, cudaMemcpyAsync(v, H->flag, 2 * sizeof(int), cudaMemcpyDeviceToHost, st), "cudaMemcpyAsync");
    CK(H, cudaStreamSynchronize(st), "cudaStreamSynchronize");
    *status_host = v[0] | v[1];
    return TF_LBM_OK;
}

int tf_lbm_get_state(tf_lbm_handle* H, void* f, void* stream)
{
    if (!H) return fail(nullptr, TF_LBM_ERR_ARG, "handle is NULL");
    int rc;
    if ((rc = check_dev_ptr(H, f, "f", false))) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e = aux_get_state(H->desc, H->buf[H->cur], (double*)f, H->G, st);
    CK(H, e, "get_state kernel");
    return TF_LBM_OK;
}

int tf_lbm_set_state(tf_lbm_handle* H, const void* f, void* stream)
{
    if (!H) return fail(nullptr, TF_LBM_ERR_ARG, "handle is NULL");
    int rc;
    if ((rc = check_dev_ptr(H, f, "f", false))) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e = aux_set_state(H->desc, H->buf[H->cur], (const double*)f, H->G, st);
    CK(H, e, "set_state kernel");
    return TF_LBM_OK;
}

int64_t tf_lbm_time(const tf_lbm_handle* H) { return H ? H->time : -1; }

int tf_lbm_get_launch(const tf_lbm_handle* H, tf_lbm_launch* out)
{
    if (!H || !out) return TF_LBM_ERR_ARG;
    out->block_x = H->shape.block_x;
    out->rows = H->shape.rows;
    out->graph_chunk = H->graph_chunk;
    out->pipeline = H->shape.pipeline;
    return TF_LBM_OK;
}

int tf_lbm_set_launch(tf_lbm_handle* H, const tf_lbm_launch* in)
{
    if (!H) return fail(nullptr, TF_LBM_ERR_ARG, "handle is NULL");
    if (!in) return fail(H, TF_LBM_ERR_ARG, "launch is NULL");
    const int bx = in->block_x;
    if (bx != 64 && bx != 128 && bx != 256) return fail(H, TF_LBM_ERR_ARG, "block_x must be 64, 128 or 256");
    if (in->rows < 1 || in->rows > 65535) return fail(H, TF_LBM_ERR_ARG, "rows must be in [1, 65535]");
    if (in->graph_chunk < 0 || (in->graph_chunk % 2) != 0 || in->graph_chunk > 4096)
        return fail(H, TF_LBM_ERR_ARG, "graph_chunk must be 0 or an even number <= 4096");
    if (in->pipeline != kPipeTma && in->pipeline != kPipeLdg && in->pipeline != kPipeAsync &&
        in->pipeline != kPipePair)
        return fail(H, TF_LBM_ERR_ARG,
                    "pipeline must be 0 (bulk copies), 1 (per-thread loads), 2 (per-thread async copies) "
                    "or 3 (two columns per thread)");
    if (in->pipeline == kPipePair && !pair_pipeline_ok(H->G.nx, H->desc.store))
        return fail(H, TF_LBM_ERR_ARG, "the two-column pipeline needs nx even and an FP32 compute type");
    if (in->pipeline == kPipeAsync && H->msize != H->esize)
        return fail(H, TF_LBM_ERR_ARG, "the async-copy pipeline needs FP32 or FP64 storage");
    if (in->pipeline == kPipeTma && !tma_pipeline_ok(H->G.nx))
        return fail(H, TF_LBM_ERR_ARG, "the bulk-copy pipeline needs nx to be a multiple of 8 and >= 16");
    drop_graphs(H);
    // the fields of the shape that init or tuning chose stand for all of it:
    // its balanced bands, and the tiles or the four-column march it runs
    if (bx == H->own.block_x && in->rows == H->own.rows && in->pipeline == H->own.pipeline) H->shape = H->own;
    else H->shape = Shape{bx, in->rows, in->pipeline};
    H->graph_chunk = in->graph_chunk;
    return TF_LBM_OK;
}

// Not part of the interface: run the tiles that block_x names (tile_of) on any
// lattice, in steps and in the handle's tapes, for the tests of tile edges.
int tflbm_use_tiles(tf_lbm_handle* H, int32_t block_x, int32_t graph_chunk)
{
    if (!H || (block_x != 64 && block_x != 128 && block_x != 256) || graph_chunk < 0 || graph_chunk % 2 != 0)
        return TF_LBM_ERR_ARG;
    drop_graphs(H);
    H->shape.tile = H->tape_tile = block_x;
    H->shape.wide = 0;
    H->graph_chunk = graph_chunk;
    return TF_LBM_OK;
}

// The same for the four-column march, over whatever march the shape describes.
int tflbm_use_wide(tf_lbm_handle* H)
{
    if (!H || H->dbl || H->p.forcing != 0 || make_consts<float>(H).omega != 1.0f || !wide_applies(H->desc.store, H->G, H->G.nx % 4 == 0))
        return TF_LBM_ERR_ARG;
    drop_graphs(H);
    H->shape.tile = 0;
    H->shape.wide = wide_bands(H->G, wide_slots(H->desc.store, H->G.nx % 4 == 0, H->sms));
    return TF_LBM_OK;
}

int tf_lbm_set_wait_limit(tf_lbm_handle* H, int32_t polls)
{
    if (!H) return fail(nullptr, TF_LBM_ERR_ARG, "handle is NULL");
    H->wait_limit = polls < 0 ? kWaitLimit : polls;
    drop_graphs(H);  // captured launches carry the old limit
    return TF_LBM_OK;
}

void tf_lbm_destroy(tf_lbm_handle* H)
{
    if (!H) return;
    cudaDeviceSynchronize();
    drop_graphs(H);
    if (H->cap) cudaStreamDestroy(H->cap);
    if (H->block) cudaFree(H->block);
    if (H->adj) cudaFree(H->adj);
    if (H->dscr) cudaFree(H->dscr);
    if (H->tscr) cudaFree(H->tscr);
    delete H;
}

}  // extern "C"
