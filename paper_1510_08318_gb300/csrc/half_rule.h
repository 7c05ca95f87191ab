// Which calls at N_p = 256 take the half-image kernels (moff_half256.cu) and which the 4-CTA clusters (host code).
#pragma once

namespace epic {

// A half image occupies one SM, an image a cluster of four; 36 clusters reside on 152 SMs (GPCs whose SMs are no
// multiple of four leave some idle).  Either form takes its items in waves, so each rule compares waves times the cost
// of one (us).  n_ent: entries of the mapping (of an item, on average), since the halves are gridded twice and the
// clusters' time grows with the longest lists of cells.  The constants are fitted to 1,529 calls of 61 to 1,024 antennas
// on footprints of 1 to 30 x 30 cells, 1 to 1,216 samples, 1 to 608 (channel, pol), FP16, for which the choice is at most
// 3 % slower than the clusters and 0.7 % slower than the better form on average (the adjoint's, FP16 and complex64: never
// slower, 0.9 %).  Some of them (us, halves and clusters):
// 331 antennas of one cell, one (channel, pol): 38 images 41 and 37, 76 images 59 and 44, 152 images 70 and 60, 342 images
// 93 and 99, 608 images 139 and 151; 152 (channel, pol) of one image 96 and 109; 271 antennas of 5 x 5 cells, 4 (channel,
// pol) of 30 images 56 and 53, 6 of 20 images 70 and 52; 331 antennas of 30 x 30 cells: 76 images 84 and 317, 608 images
// 376 and 1,701.  The adjoint, one cell: 38 images 35 and 40, 76 images 36 and 55, 608 images 184 and 264; 7 x 7 cells:
// 160 images 107 and 102, 608 images 260 and 320.
inline long long half_waves(long long n_items, int n_sm) { return (2 * n_items + n_sm - 1) / n_sm; }
inline long long resident_clusters(int n_sm) { return 9LL * n_sm / 38 > 0 ? 9LL * n_sm / 38 : 1; }
inline long long cluster_waves(long long n_items, int n_sm) {
    return (n_items + resident_clusters(n_sm) - 1) / resident_clusters(n_sm);
}

// Sums that the worker with most of them adds to the accumulators, where n_work workers share `units` units in order, and
// every `run` units belong to the same sums: worker w has the units from units w / n_work (rounded down) on.
inline long long most_sums(long long units, long long n_work, long long run) {
    if (n_work > units) n_work = units;
    const long long share = (units + n_work - 1) / n_work;
    bool even = share > run ? units % n_work == 0 && share % run == 0 : true;   // every sum begins with a worker
    if (share <= run)
        for (long long b = run; even && b < units; b += run) even = units * ((b * n_work + units - 1) / units) / n_work == b;
    return even ? (share + run - 1) / run : share < 2 ? 1 : (share - 2) / run + 2;
}

// Forward.  Adding sums to the accumulators takes 12 us a half image and 6 us an image.  Where the waves of halves are
// full their CTAs end together, and the additions wait for each other, most of all those to one (channel, pol) of n_cp.
inline bool half_pays_fwd(long long n_items, int n_sm, double n_ent, long long n_cp) {
    const long long run = n_cp > 0 && n_items > n_cp ? n_items / n_cp : 1;
    const double wh = double(half_waves(n_items, n_sm)), wc = double(cluster_waves(n_items, n_sm));
    const double sh = double(most_sums(2 * n_items, n_sm, run)), sc = double(most_sums(n_items, resident_clusters(n_sm), run));
    const double fill = 2.0 * double(n_items) / (wh * n_sm);
    return 3.0 + (12.0 + 10.0 / double(n_cp)) * fill + 12.0 * (sh - 1.0) + wh * (13.0 + 8e-5 * n_ent) <=
           6.0 * (sc - 1.0) + wc * (7.6 + 6e-5 * n_ent + 8e-10 * n_ent * n_ent);
}

// Adjoint (its sums are one complex number per antenna).
inline bool half_pays_bwd(long long n_items, int n_sm, double n_ent) {
    return half_waves(n_items, n_sm) * (23.0 + 1e-3 * n_ent) <= cluster_waves(n_items, n_sm) * (14.0 + 4.5e-4 * n_ent);
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
