// Instantiation of the forward and adjoint MOFF kernels for N_p = 256.
#include "half_rule.h"
#include "moff_fwd.cuh"
#include "moff_bwd.cuh"

namespace epic {

// Which form.  The half-image kernels (moff_half256.cu) need every plan of the launch to have their table (up to
// 1,471 antennas); the 4-CTA clusters take more antennas, the cross-polarisation products, a batch's request for one
// row-pass buffer, and the calls for which they are the faster form (half_rule.h).
static bool all_half(const SegList& L) {
    for (int s = 0; s < L.n_seg; ++s)
        if (!L.seg[s].half.run) return false;
    return true;
}

static cudaError_t launch_clusters(int vdt, const SegList& L, int n_sm, cudaStream_t st, bool xpol) {
    switch (vdt) {
        case 0: return xpol ? launch_fwd_t<256, 0, true>(L, n_sm, st) : launch_fwd_t<256, 0>(L, n_sm, st);
        case 1: return xpol ? launch_fwd_t<256, 1, true>(L, n_sm, st) : launch_fwd_t<256, 1>(L, n_sm, st);
        case 2: return xpol ? launch_fwd_t<256, 2, true>(L, n_sm, st) : launch_fwd_t<256, 2>(L, n_sm, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_fwd_256(int vdt, const SegList& L, int n_sm, cudaStream_t st, bool xpol) {
    const long long n_items = L.first[L.n_seg];
    if (xpol || n_items == 0 || !all_half(L)) return launch_clusters(vdt, L, n_sm, st, xpol);
    double n_ent = 0.0;
    long long n_cp = 0;
    for (int s = 0; s < L.n_seg; ++s) {
        n_ent += double(L.seg[s].half.n_ent) * double(L.first[s + 1] - L.first[s]) / double(n_items);
        n_cp += L.seg[s].n_cp;
    }
    const HalfChoice form = half_choice(n_items, n_sm, n_ent, n_cp, L.max_workers, L.max_buffers == 1);
    if (form.cap == L.max_workers)
        return form.half ? launch_half256_fwd(vdt, L, n_sm, st) : launch_clusters(vdt, L, n_sm, st, xpol);
    SegList capped = L;
    capped.max_workers = form.cap;
    return launch_clusters(vdt, capped, n_sm, st, xpol);
}

cudaError_t launch_bwd_256(int vdt, const BwdArgs& a, int n_sm, cudaStream_t st) {
    if (a.half.run && half_pays_bwd(a.n_items, n_sm, a.half.n_ent)) return launch_half256_bwd(vdt, a, n_sm, st);
    switch (vdt) {
        case 0: return launch_bwd_t<256, 0>(a, n_sm, st);
        case 1: return launch_bwd_t<256, 1>(a, n_sm, st);
        case 2: return launch_bwd_t<256, 2>(a, n_sm, st);
        default: return cudaErrorInvalidValue;
    }
}

// SMs where the antennas fit the half images (half_choice turns a cap into clusters), else clusters.
int resident_fwd_workers_256(int vdt, int max_ant, int n_sm) {
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess &&
        half256_fits(max_ant, (size_t)optin))
        return n_sm;
    switch (vdt) {
        case 0: return resident_fwd_workers_t<256, 0>(max_ant, n_sm);
        case 1: return resident_fwd_workers_t<256, 1>(max_ant, n_sm);
        case 2: return resident_fwd_workers_t<256, 2>(max_ant, n_sm);
        default: return 0;
    }
}

}  // namespace epic
