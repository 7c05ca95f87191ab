// Instantiation of the forward and adjoint MOFF kernels for N_p = 256.
#include "moff_fwd.cuh"
#include "moff_bwd.cuh"

namespace epic {

// Which form.  The half-image kernels (moff_half256.cu) need every plan of the launch to have their table (up to
// 1,471 antennas); the 4-CTA clusters take more antennas, the cross-polarisation products, a batch's request for one
// row-pass buffer, and calls of few images, where a cluster finishes an image sooner than two SMs their halves.
// Measured: a half image takes an SM 14.5 us and an image a cluster 7.8 us (331 antennas, 7.05 against 6.05 ms for
// 32,768 images); the adjoint 33 and 20 us (1,024 antennas).  So the line lies where the waves of half
// images over the SMs take less time than the waves of images over n_sm / 4 clusters.
static bool half_pays(long long n_items, int n_sm, int half_cost, int cluster_cost) {
    const long long n_cl = n_sm / 4 > 0 ? n_sm / 4 : 1;
    return (2 * n_items + n_sm - 1) / n_sm * half_cost <= (n_items + n_cl - 1) / n_cl * cluster_cost;
}

static bool use_half(const SegList& L, bool xpol, int n_sm) {
    if (xpol || L.max_buffers == 1 || L.first[L.n_seg] >= 1 << 30) return false;   // half images in 32 bits
    for (int s = 0; s < L.n_seg; ++s)
        if (!L.seg[s].half.run) return false;
    return half_pays(L.first[L.n_seg], n_sm, 15, 8);
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
    if (a.half.run && half_pays(a.n_items, n_sm, 33, 20)) return launch_half256_bwd(vdt, a, n_sm, st);
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
