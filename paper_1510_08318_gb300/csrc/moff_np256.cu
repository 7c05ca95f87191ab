// Instantiation of the forward and adjoint MOFF kernels for N_p = 256.
#include "half_rule.h"
#include "moff_fwd.cuh"
#include "moff_bwd.cuh"

namespace epic {

// Which form.  The half-image kernels (moff_half256.cu) need every plan of the launch to have their table (up to
// 1,471 antennas); the 4-CTA clusters take more antennas, the cross-polarisation products, a batch's request for one
// row-pass buffer, and the calls for which they are the faster form (half_rule.h).
static bool use_half(const SegList& L, bool xpol, int n_sm) {
    const long long n_items = L.first[L.n_seg];
    if (xpol || L.max_buffers == 1 || n_items < 1 || n_items >= 1 << 30) return false;   // half images in 32 bits
    double n_ent = 0.0;
    long long n_cp = 0;
    for (int s = 0; s < L.n_seg; ++s) {
        if (!L.seg[s].half.run) return false;
        n_ent += double(L.seg[s].half.n_ent) * double(L.first[s + 1] - L.first[s]) / double(n_items);
        n_cp += L.seg[s].n_cp;
    }
    return half_pays_fwd(n_items, n_sm, n_ent, n_cp);
}

cudaError_t launch_fwd_256(int vdt, const SegList& L, int n_sm, cudaStream_t st, bool xpol) {
    if (use_half(L, xpol, n_sm)) return launch_half256_fwd(vdt, L, n_sm, st);
    switch (vdt) {
        case 0: return xpol ? launch_fwd_t<256, 0, true>(L, n_sm, st) : launch_fwd_t<256, 0>(L, n_sm, st);
        case 1: return xpol ? launch_fwd_t<256, 1, true>(L, n_sm, st) : launch_fwd_t<256, 1>(L, n_sm, st);
        case 2: return xpol ? launch_fwd_t<256, 2, true>(L, n_sm, st) : launch_fwd_t<256, 2>(L, n_sm, st);
        default: return cudaErrorInvalidValue;
    }
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
