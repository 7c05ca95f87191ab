// Rules by which launches choose between kernel variants (host code; each with the measurements behind its line).
#pragma once
#include <cstddef>

namespace epic {

// X-engine, voltages read one by one (FP16, or 4+4 bits that 4-byte loads don't fit): whether an integration is so
// short that the blocks' epilogues take longer than their decode.  It then takes two decode sets and 8 epilogue warps,
// else three and 4.  Measured (us, short and long form, 256 (channel, pol) where not said otherwise, 152 SMs): FP16, 256
// antennas: 96 samples 47 and 65, 256 samples 65 and 78, 512 samples 103 and 104, 1,024 samples 185 and 183.  4+4 bits: 130
// antennas 64 samples 27 and 31, 128 samples 37 and 39, 1,024 samples 213 and 168; 254 antennas 128 samples 57 and 72, 256
// samples 90 and 83.
inline bool xeng_short(bool fp16, int n_time) { return n_time <= (fp16 ? 768 : 224); }

// FX imaging: planes per group of the lag gather.  Narrow groups keep more of a tile's pairs in L1 and give more CTAs,
// wide ones read each table entry and its row of visibilities fewer times.  Measured (us; 256 antennas, N_p = 128, 160
// entries a lag cell) with 2, 4, 8, 16, 32 planes per group: 4 planes 64, 68, 78, -, -; 8 planes 88, 72, 81, 107, -; 16
// planes 167, 99, 89, 108, 171; 32 planes 310, 170, 107, 109, 181; 64 planes 616, 333, 198, 141, 189; 128 planes -, -,
// 367, 252, 229.  Few antennas leave few entries to a lag cell (48 of 5 x 5 cells at N_p = 128: 6), and the CTAs
// themselves set the time: one group, up to 32 planes, as far as the tiles alone fill the SMs.  Measured (us; 48
// antennas) with the widths above and with one group: 5 planes 35 and 29, 8 planes 33 and 30, 33 planes 49 and 41, 64
// planes 46 and 39; 100 antennas (25 entries a cell) 5 planes 39 and 35, 8 planes 34 and 33, 16 planes 37 and 37; at N_p =
// 64 (64 tiles) 64 antennas of 3 x 3 cells 5 planes 23 and 25.
inline int fx_planes_per_group(int n_cp, int n_pad, long long n_ent) {
    if (n_pad >= 128 && n_ent < 16LL * n_pad * n_pad) {
        int g = n_cp == 1 ? 1 : 2;
        while (g < n_cp && g < 32) g *= 2;
        return g;
    }
    return n_cp >= 96 ? 32 : n_cp >= 40 ? 16 : n_cp >= 12 ? 8 : n_cp >= 6 ? 4 : n_cp >= 2 ? 2 : 1;
}

// Auto-correlation term: CTAs of a (channel, pol)'s cluster (kAcThreads = 512 threads each, at least two antennas and 512
// pixels).  The CTAs share the antennas' sum and the pixels, but each does the first half of the transform, and past
// what the SMs hold at once they come in waves: the least waves times (share done by each + rest / CTAs).  Clusters of
// 4 and 8 leave some SMs of a GPC idle.  Measured (us a call of one sample; 1, 2, 4, 8 CTAs): 400 antennas of 15 x 15
// cells, N_p = 512, one CTA an SM: 16 (channel, pol) 812, 487, 306, 339; 64: 1151, 741, 775, 963; 150: 1456, 1489, 1828,
// 1962; 200: 2475, 2120, 2258, 2664; 331 antennas of 7 x 7 cells, N_p = 256, four an SM: 64: 165, 115, 103, 107; 150: 259,
// 208, 223, 227; 400: 554, 538, 535, 579.
inline int autocorr_cluster(long long n_cp, int n_ant, int n_pad, int lag_side, size_t smem, int n_sm) {
    const long long fit = (long long)(228 * 1024 / (smem + 1024)), per_sm = fit < 1 ? 1 : fit > 4 ? 4 : fit;
    // lags x pixels of a row in the first half of the transform; those of the whole image in the second
    const double each = 0.05 + double(lag_side) / (lag_side + n_pad);
    int best = 1;
    double least = 0.0;
    for (int n_cl = 1; n_cl <= 8 && (n_cl == 1 || (2 * n_cl <= n_ant && n_pad * n_pad >= 512 * n_cl)); n_cl *= 2) {
        const long long held = n_sm * per_sm * (n_cl == 8 ? 28 : n_cl == 4 ? 36 : 38) / 38 / n_cl;
        const double cost = double((n_cp + held - 1) / (held > 0 ? held : 1)) * (each + (1.0 - each) / n_cl);
        if (n_cl == 1 || cost < least) best = n_cl, least = cost;
    }
    return best;
}

}  // namespace epic
