// Internal definition of the opaque tf_lbm_handle, shared by the C-ABI
// translation units (tflbm_api.cu, tflbm_adjoint.cu).  Not part of the ABI.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include "../../include/tflbm.h"
#include "tflbm_internal.h"

using namespace tflbm;

struct tf_lbm_handle {
    tf_lbm_params p;
    int device = 0;
    int sms = 152;             // streaming multiprocessors of the device
    size_t esize = 4;          // bytes of the compute type (plane 0, fields)
    size_t msize = 4;          // bytes of one stored moving population
    bool dbl = false;          // compute type is double
    StoreDesc desc{};          // storage encoding (for the auxiliary kernels)
    Geom G{};
    void* block = nullptr;     // one allocation for everything below that is not lazy
    void* buf[2] = {nullptr, nullptr};
    int cur = 0;               // buf[cur] holds the post-collision populations of step t-1
    void* kappa = nullptr;     // [ny][nx] or null (uniform)
    double kappa_u = 0.0;
    double href = 0.0;         // reference height (exactly representable in the storage type)
    double* partials = nullptr;
    double* result = nullptr;
    int nmass = 0;
    int* flag = nullptr;
    int* status = nullptr;     // device word kernels set (kStatusTimeout)
    int wait_limit = kWaitLimit;  // polls of one mbarrier before a bulk-copy kernel gives up
    int64_t time = 0;
    Shape shape{128, 64, kPipeLdg};  // replaced by the occupancy-derived default in tf_lbm_init
    Shape def{128, 64, kPipeLdg};    // the default: what tuning puts tiles and the four-column march on
    Shape own{128, 64, kPipeLdg};    // what init or tuning chose: setting its fields gives it back whole
    Shape one{128, 64, kPipePair};   // the two-column march that takes a run of one FP32 step of a wide shape
    int tape_tile = 0;               // tests: block_x of a tape's tiles, forward and adjoint; 0: by the lattice
    int graph_chunk = 0;
    cudaStream_t cap = nullptr;
    cudaGraphExec_t exec[2] = {nullptr, nullptr};
    std::string err;
    void* adj = nullptr;       // adjoint scratch (lazy): 10 fields of the compute type
    void* dscr = nullptr;      // diagnostics scratch (lazy): one BatchDomain entry + partial sums + trig table
    void* tscr = nullptr;      // term-norm scratch (lazy): 5 fields + partial sums
};


namespace tflbm {
// Offsets of several arrays in one allocation, each on a 256-byte boundary.
struct Carver {
    size_t total = 0;
    size_t take(size_t bytes)
    {
        const size_t at = total;
        total += (bytes + 255) / 256 * 256;
        return at;
    }
};
// Per-run step constants of a handle, in the compute type T.
template <typename T>
Consts<T> make_consts(const tf_lbm_handle* H);
// Launch one fused step from buf[from] into buf[from ^ 1].  A run of steps marks
// its first and last one: between two steps of a run the buffer may hold
// moments instead of populations (Shape::wide).
cudaError_t launch_one_step(tf_lbm_handle* H, int from, cudaStream_t st, bool first = true, bool last = true);
// One tile step between two population buffers of the handle's layout that
// also records the moments of the state it starts from (tflbm_tile.cuh).
cudaError_t launch_recorded_step(tf_lbm_handle* H, const void* fin, void* fout, void* mom, cudaStream_t st);
// block_x of the tile kernel for a lattice (see tile_of), forward and adjoint.
int tile_block_x(int store, int nx, int ny, int sms, bool omega1);
int adjoint_block_x(bool dbl, int nx, int ny, int sms);
// Record an error message on H (or for the calling thread when H is null).
int handle_fail(tf_lbm_handle* H, int code, const std::string& msg);
int handle_cuda_fail(tf_lbm_handle* H, cudaError_t e, const char* what);
// ARG error unless ptr is device or managed memory of the current device.
int handle_check_dev_ptr(tf_lbm_handle* H, const void* ptr, const char* name, bool allow_null);
// Forget the handle's captured step graphs (after a launch-shape change).
void handle_drop_graphs(tf_lbm_handle* H);
// Adjoint of one step (tflbm_adjoint.cu).
cudaError_t adjoint_step_dispatch(tf_lbm_handle* H, const void* f, const void* a_next, void* a,
                                  void* grad_kappa, cudaStream_t st);
}  // namespace tflbm
