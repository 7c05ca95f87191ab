// Rules by which launches choose between kernel variants (host code; each with the measurements behind its line).
#pragma once

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

}  // namespace epic
