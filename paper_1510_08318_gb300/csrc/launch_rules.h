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

}  // namespace epic
