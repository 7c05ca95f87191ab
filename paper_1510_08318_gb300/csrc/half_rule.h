// Which calls at N_p = 256 take the half-image kernels (moff_half256.cu) and which the 4-CTA clusters (host code).
#pragma once

namespace epic {

// A half image occupies one SM, an image a cluster of four; 36 clusters reside on 152 SMs (GPCs whose SMs are no
// multiple of four leave some idle).  Either form takes its items in waves, so each rule compares waves times the cost
// of one (us).  n_ent: entries of the mapping (of an item, on average), since the halves are gridded twice and the
// clusters' time grows with the longest lists of cells.  The constants are fitted to calls of 331 and 1,024 antennas on
// footprints of 1 to 30 x 30 cells, 1 to 1,216 samples, 1 to 608 (channel, pol), FP16.  Some of them (us, halves and
// clusters): 331 antennas of one cell, one (channel, pol): 38 images 41 and 37, 76 images 59 and 44, 152 images 70 and
// 60, 342 images 93 and 99, 608 images 139 and 151; 152 (channel, pol) of one image 96 and 109; 331 antennas of 30 x 30
// cells: 76 images 84 and 317, 608 images 376 and 1,701.  The adjoint, one cell: 38 images 35 and 40, 76 images 36 and
// 55, 608 images 184 and 264; 7 x 7 cells: 160 images 107 and 102, 608 images 260 and 320.
inline long long half_waves(long long n_items, int n_sm) { return (2 * n_items + n_sm - 1) / n_sm; }
inline long long cluster_waves(long long n_items, int n_sm) {
    const long long n_cl = 9LL * n_sm / 38 > 0 ? 9LL * n_sm / 38 : 1;
    return (n_items + n_cl - 1) / n_cl;
}

// Forward.  Where the waves of halves are full their CTAs end together, and the additions of their sums to the few
// accumulators of n_cp (channel, pol) wait for each other: 22 us for one.
inline bool half_pays_fwd(long long n_items, int n_sm, double n_ent, long long n_cp) {
    const double wh = double(half_waves(n_items, n_sm)), wc = double(cluster_waves(n_items, n_sm));
    const double fill = 2.0 * double(n_items) / (wh * n_sm);
    return 22.0 * fill / double(n_cp) + wh * (13.5 + 8e-5 * n_ent) <= wc * (7.7 + 6e-5 * n_ent + 6e-10 * n_ent * n_ent);
}

// Adjoint (its sums are one complex number per antenna).
inline bool half_pays_bwd(long long n_items, int n_sm, double n_ent) {
    return half_waves(n_items, n_sm) * (23.0 + 8e-4 * n_ent) <= cluster_waves(n_items, n_sm) * (15.0 + 4e-4 * n_ent);
}

// The form of a forward launch whose plans all have their half images, and the cap on its CTAs or clusters (0: none).
// A launch is capped in SMs (max_workers, 0: none), since the caller does not know the form: a cluster stands for four.
struct HalfChoice {
    bool half;
    int cap;
};
inline HalfChoice half_choice(long long n_items, int n_sm, double n_ent, long long n_cp, int max_workers, bool one_buffer) {
    const int sms = max_workers > 0 && max_workers < n_sm ? max_workers : n_sm;
    // half images are numbered in 32 bits
    if (!one_buffer && n_items < 1 << 30 && half_pays_fwd(n_items, sms, n_ent, n_cp)) return {true, max_workers};
    return {false, max_workers > 0 ? (sms / 4 > 0 ? sms / 4 : 1) : 0};
}

}  // namespace epic
