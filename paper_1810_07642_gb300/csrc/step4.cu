// Launches of the four-column march (tflbm_step4.cuh) per storage type.
#include <algorithm>

#include "tflbm_step4.cuh"

namespace tflbm {

namespace {

// Calls fn with the kernel's template arguments as types: storage, moments in
// and out, nx a multiple of 4.
template <typename Fn>
cudaError_t wide_variant(int store, bool mom_in, bool mom_out, bool quad, Fn fn)
{
    using Y = std::true_type;
    using N = std::false_type;
    if (store == kStoreF32) {
        if (mom_in && mom_out) return quad ? fn(float(), Y(), Y(), Y()) : fn(float(), Y(), Y(), N());
        if (mom_in) return quad ? fn(float(), Y(), N(), Y()) : fn(float(), Y(), N(), N());
        if (mom_out) return quad ? fn(float(), N(), Y(), Y()) : fn(float(), N(), Y(), N());
        return cudaErrorInvalidValue;  // a run of one step has other kernels
    }
    if (mom_in || mom_out || !quad) return cudaErrorInvalidValue;
    if (store == kStoreF16) return fn(__half(), N(), N(), Y());
    if (store == kStoreBF16) return fn(__nv_bfloat16(), N(), N(), Y());
    return cudaErrorInvalidValue;
}

}  // namespace

bool wide_applies(int store, const Geom& G, bool quad)
{
    if (store == kStoreF64) return false;
    if (quad) return G.nx % 4 == 0;
    return store == kStoreF32 && G.nx >= 8 && 6LL * mom_pitch(G.nx) * G.ny + 128 <= 9LL * G.plane;
}

int wide_strips(int nx) { return (nx + kWideCols - 1) / kWideCols; }

cudaError_t launch_wide(int store, bool mom_in, bool mom_out, const void* fin, void* fout, const void* kappa,
                        const Geom& G, const Consts<float>& C, int bands, cudaStream_t st)
{
    return wide_variant(store, mom_in, mom_out, G.nx % 4 == 0, [&](auto sm, auto mi, auto mo, auto q) {
        return launch_dependent(k_step4<decltype(sm), decltype(mi)::value, decltype(mo)::value, decltype(q)::value>,
                                dim3(wide_strips(G.nx), bands), 32, 0, st, fin, fout, (const float*)kappa, G, C);
    });
}

cudaError_t launch_wide_batch(int store, bool mom_in, bool mom_out, const BatchItem* items, int nitems,
                              const void* doms, int parity, cudaStream_t st)
{
    return wide_variant(store, mom_in, mom_out, true, [&](auto sm, auto mi, auto mo, auto) {
        return launch_dependent(k_step4_batch<decltype(sm), decltype(mi)::value, decltype(mo)::value>, dim3(nitems), 32,
                                0, st, items, (const BatchDomain<float>*)doms, parity);
    });
}

int wide_slots(int store, bool quad, int sms)
{
    int occ = 0;
    const bool f32 = store == kStoreF32;
    const cudaError_t e = wide_variant(store, f32, f32, quad, [&](auto sm, auto mi, auto mo, auto q) {
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &occ, k_step4<decltype(sm), decltype(mi)::value, decltype(mo)::value, decltype(q)::value>, 32, 0);
    });
    if (e != cudaSuccess) {
        cudaGetLastError();
        occ = 0;
    }
    return std::max(occ, 1) * sms;
}

}  // namespace tflbm
