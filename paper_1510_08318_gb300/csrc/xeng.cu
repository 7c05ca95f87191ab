// X-engine of the FX route (Sec. 3 "FX" flow; Eq. "cc-vis"): the visibilities
//   V_ab = g_a conj(g_b) (1/T) sum_t V_a(t) conj(V_b(t))
// of every antenna pair of every (channel, pol), as a Hermitian product E E^H on the
// 5th-generation tensor cores.
//
// Per (channel, pol) the voltages form E [A x T] complex; with R = Re E and I = Im E
//   Re V = R_a R_b^T + I_a I_b^T,   Im V = I_a R_b^T - R_a I_b^T   (summed over t),
// four real products with K = T.  4+4-bit and FP16 voltages are exact in FP16, and each product
// (at most 64 in magnitude for 4+4-bit) is accumulated in FP32 exactly while the sums stay below
// 2^24, so the raw sums are exact.
//
// Work unit: a 128 x 128 block (antenna rows a in block ab, columns b in block bb, bb >= ab:
// the upper block triangle, the lower one follows by Hermitian symmetry) of one (channel,
// pol); one persistent CTA per SM takes a contiguous range of units, K walked in chunks of 32
// samples.  A chunk's operands are K-major FP16 planes: the B tile [R_b; I_b; -R_b] (384 rows)
// and the A tile [R_a; I_a] (a diagonal unit takes its A planes from the B tile), so that two
// MMAs with N = 256 per 16 samples give D = R_a [R_b; I_b]^T + I_a [I_b; -R_b]^T (without the plane -R_b
// where voltages are read one by one: two MMAs of N = 128, one with its A operand negated, for the second):
// Re V in columns 0..127 and -Im V in 128..255.  The CTA's warps have three roles, handing work
// over through mbarriers only (no CTA-wide barrier inside the loop):
//   - sets of 8 decode warps (two, or three for long integrations read one by one) take the chunks in turn and
//     convert their voltages (loaded into registers three of the set's chunks ahead) into one
//     stage of a 3-stage ring; each warp fences
//     its stores for the tensor cores and arrives on the stage's full barrier, and refills a
//     stage after the MMAs that read it have completed (the stage's empty barrier, signalled by
//     tcgen05.commit);
//   - one thread of the MMA warp issues the MMAs (M = 128, K = 16) of a chunk into one
//     of two TMEM accumulator buffers (all 512 columns), commits each chunk to its stage's empty
//     barrier and a unit's last chunk to the buffer's full barrier;
//   - 8 (or 4) epilogue warps read a finished buffer (tcgen05.ld), scale by g_a conj(g_b) / T with
//     the gains in shared memory, write the block (16 adjacent elements at a time) and, off the
//     diagonal, its mirrored conjugate, then release the buffer, while the next unit fills the
//     other one.
// Every wait is bounded by the plan's try count and taken by a whole warp; on a timeout the role
// stops, the CTA sets the correlator-timeout bit of the plan's status word and writes NaN into
// its first output element; the MMA warp waits (full limit) for the MMAs it issued before the
// tensor memory is released.
//
// WIDE (4+4-bit voltages, A a multiple of 4, 4-byte aligned input): a thread loads 4 antennas
// of each of its 8 samples with 4-byte loads (a warp reads whole 128-byte rows), transposes the
// 4 x 4 byte blocks with byte permutes and converts each 4 samples of an antenna with two
// permute + packed-subtraction pairs per plane.  Other voltages are read one by one.
//
// Bound by the latency of the decode's loads and of the epilogue's stores (the products alone take 43 us of
// 115 in the first case below) and, where the units do not divide over the SMs, by the last of them (768 units on
// 152 SMs: six turns for 5.05).  A copy of the kernel without the epilogue's 15 / 16 took 72 of 105 us: its
// column gains came from L2 one by one, because the stages leave a few KB of the SM to L1.  Measured before and
// now (us; antennas x samples x (channel, pol)): 4+4-bit 256 x 1024 x 256: 140 and 116; 256 x 64 x 256: 88 and 44;
// 256 x 1024 x 1: 37 and 29; 1024 x 1024 x 16: 111 and 95; 254 x 1024 x 256: 287 and 239; FP16 256 x 1024 x 256: 292
// and 182.
#include <algorithm>
#include <cuda_fp16.h>
#include <cstdint>
#include "launch_rules.h"
#include "moff_common.cuh"
#include "tcgen05.cuh"

namespace epic {
namespace xe {
using namespace tc;

constexpr int TC = 32;                      // samples per K chunk (K = 32: one real plane per operand row)
// K-major FP16 planes without swizzle: 8 x 8 core matrices of 128 bytes, a row group of 8 rows
// holding the chunk's 4 core matrices along K
constexpr int kRowGroupBytes = 4 * 128;
constexpr int kPlaneBytes = 16 * kRowGroupBytes;       // 128 rows x 32 samples (8 KB)
constexpr int kATileBytes = 2 * kPlaneBytes;           // [Re_a; Im_a]
constexpr uint32_t kNegA = 1u << 13;                   // instruction descriptor: negate the A operand
// an epilogue warp's 32 rows x 16 columns, rows 144 bytes apart (16-byte accesses of 8 lanes hit all 32 banks)
constexpr int kRowStride = 18;

// The roles of a CTA's warps (one CTA per SM).  Measured (us, 256 antennas, 256 (channel, pol), 4+4-bit voltages of
// 1,024 and of 64 samples; sets, epilogue warps, stages): 2, 8, 3: 116 and 44; 3, 4, 3: 113 and 61; 2, 8, 4: 121 and
// 45; 3, 4, 5: 119 and 61; 1, 8, 4: 193 and 54.  More stages leave less L1 for the loads in flight: FP16 voltages of
// 1,024 samples (read one by one, with three sets) take 192 with 3 stages and 257 with 5.  SHORT: the roles of a
// short integration of voltages read one by one (xeng_short).
template <bool WIDE, bool SHORT>
struct Roles {
    static constexpr int NDS = WIDE || SHORT ? 2 : 3;       // decode warp sets, taking alternate chunks
    static constexpr int NDW = 8 * NDS;                     // decode warps (a set's tile mappings take 256 threads)
    static constexpr int NEW = WIDE || SHORT ? 8 : 4;       // epilogue warps, NEW / 4 per TMEM lane quarter
    static constexpr int MMA_WARP = NDW;                    // the warp whose first thread issues the MMAs
    static constexpr int NT = 32 * (NDW + 1 + NEW);
    // the B tile with the plane -Re_b, or without: then its product is one MMA of N = 128 more with the A operand
    // negated.  Without it the decode stores a plane less, and the MMAs read their operands in smaller pieces.
    // Measured (us, with and without, 256 antennas, 256 (channel, pol), 1,024 samples): 4+4-bit 116.9 and 117.6, one
    // (channel, pol) 29.2 and 30.0; FP16 192 and 182, 254 antennas of 4+4 bits 254 and 239.
    static constexpr bool NEG_PLANE = WIDE;
    static constexpr int kBTileBytes = (NEG_PLANE ? 3 : 2) * kPlaneBytes;   // [Re_b; Im_b; -Re_b] or [Re_b; Im_b]
    static constexpr int kStageBytes = kBTileBytes + kATileBytes;           // 40 or 32 KB
    static constexpr int NSTAGE = 3;
    // a set waits for its stage's last use but one at most: with fewer stages than sets it could take the phase
    // before for the one it waits for
    static_assert(NSTAGE >= NDS, "stages");
    // mbarriers: stage full [NSTAGE], stage empty [NSTAGE], accumulator full [2], accumulator
    // empty [2], drain
    static constexpr int N_MBAR = 2 * NSTAGE + 5;
    static constexpr size_t kSmem = (size_t)NSTAGE * kStageBytes + (size_t)NEW * (32 * kRowStride + 128) * sizeof(float2) +
                                    8 * N_MBAR + 16;
};

// One voltage as an FP16 (re, im) pair (half2 bits).  FP16 input is already the pair.  A
// 4+4-bit byte holds two 4-bit two's-complement values (re in the high nibble); XOR with 8 biases
// each to n + 8 in [0, 15], which placed in the mantissa of 1024 (bits 0x6400 | (n + 8)) is
// exactly 1032 + n, so one packed subtraction of 1032 yields both components exactly.
template <int VDT>
__device__ __forceinline__ uint32_t voltage_pair(typename Volt<VDT>::T raw) {
    if constexpr (VDT == 1) {
        return raw;
    } else {
        const uint32_t t = (uint32_t)raw ^ 0x88u;
        const uint32_t u = ((t >> 4) & 0xFu) | ((t & 0xFu) << 16) | 0x64006400u;
        const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&u), __halves2half2(__ushort_as_half(0x6408),
                                                                                          __ushort_as_half(0x6408)));
        return *reinterpret_cast<const uint32_t*>(&h);
    }
}

// unit -> (cp, row block, column block), column block >= row block (32-bit: the launcher
// checks that the units fit)
__device__ __forceinline__ void unit_coords(int u, int nab, int& cp, int& ab, int& bb) {
    const int upc = nab * (nab + 1) / 2;
    cp = u / upc;
    int r = u - cp * upc;
    ab = 0;
    while (r >= nab - ab) {
        r -= nab - ab;
        ++ab;
    }
    bb = ab + r;
}

template <int VDT, bool WIDE, bool SHORT>
__global__ void __launch_bounds__(Roles<WIDE, SHORT>::NT, 1) xeng_kernel(const XengArgs a) {
    using W = Roles<WIDE, SHORT>;
    constexpr int NDS = W::NDS, NDW = W::NDW, NEW = W::NEW, MMA_WARP = W::MMA_WARP, NSTAGE = W::NSTAGE, N_MBAR = W::N_MBAR;
    constexpr int kBTileBytes = W::kBTileBytes, kStageBytes = W::kStageBytes;
    static_assert(!WIDE || VDT == 2, "the wide loads are for 4+4-bit voltages");
    using VT = typename Volt<VDT>::T;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* sT = smem_raw;                                               // [NSTAGE] stages
    float2* sRows = reinterpret_cast<float2*>(sT + (size_t)NSTAGE * kStageBytes);      // [NEW][32][kRowStride]
    float2* sGain = sRows + NEW * 32 * kRowStride;                                     // [NEW][128]
    uint64_t* mbar = reinterpret_cast<uint64_t*>(sGain + NEW * 128);                  // [N_MBAR]
    uint32_t* tslot = reinterpret_cast<uint32_t*>(mbar + N_MBAR);
    int* s_fail = reinterpret_cast<int*>(tslot + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int A = a.n_ant, T = a.n_time, CP = a.n_cp;
    const int nab = (A + 127) / 128;
    const int n_units = CP * (nab * (nab + 1) / 2);
    const int n_chunks = (T + TC - 1) / TC;
    const VT* V = static_cast<const VT*>(a.volt);
    auto mb_full = [&](int s) { return smem_u32(&mbar[s]); };
    auto mb_empty = [&](int s) { return smem_u32(&mbar[NSTAGE + s]); };
    auto mb_accf = [&](int b) { return smem_u32(&mbar[2 * NSTAGE + b]); };
    auto mb_acce = [&](int b) { return smem_u32(&mbar[2 * NSTAGE + 2 + b]); };
    const uint32_t mb_drain = smem_u32(&mbar[2 * NSTAGE + 4]);
    // a bounded wait taken by a whole warp: the warp goes on only if every lane saw the phase
    auto warp_wait = [&](uint32_t mb, int parity) -> bool {
        return __all_sync(0xffffffffu, mbar_wait(mb, (uint32_t)parity, a.wait_tries)) != 0;
    };

    if (tid == 0) {
        for (int s = 0; s < NSTAGE; ++s) {
            mbar_init(mb_full(s), 8);
            mbar_init(mb_empty(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(mb_accf(b), 1);
            mbar_init(mb_acce(b), NEW);
        }
        mbar_init(mb_drain, 1);
        *s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(tslot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tslot;             // accumulator buffer b: columns 256 b (Re), 256 b + 128 (Im)

    long long beg_l, end_l;
    work_range(n_units, blockIdx.x, gridDim.x, beg_l, end_l);
    const int beg = (int)beg_l, end = (int)end_l;

    if (warp < NDW) {
        // ---------------- decode warps: raw voltages -> FP16 operand planes of stage g % NSTAGE ----
        // Set dset decodes the CTA's chunks g = dset, dset + NDS, ...  Within a set, warps 0-3 fill
        // the B tile ([Re; Im; -Re] of the column block) and warps 4-7 the A tile ([Re; Im] of the
        // row block; nothing on a diagonal unit), warp dw taking samples 8 (dw % 4) .. + 7 of the
        // chunk and lane l antennas 4 l .. 4 l + 3 of the block.  The thread's slot i holds antenna
        // 4 l + (i + rot) % 4, rot = (l / 2) % 4, so that the 8 lanes of a quarter-warp write the
        // 16-byte rows of 8 distinct rows mod 8 (all 32 banks) with each 16-byte store.
        const int dw = warp & 7, dset = warp >> 3;
        const bool bside = dw < 4;
        const int so = dw & 3, rot = (lane >> 1) & 3;
        int soff[4];                                   // byte offset in a plane of slot i's row
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = 4 * lane + ((i + rot) & 3);
            soff[i] = (r >> 3) * kRowGroupBytes + so * 128 + (r & 7) * 16;
        }
        // (unit, chunk) cursors step NDS chunks at a time; true when the unit changed
        auto advance = [&](int& uu, int& kk, int by) -> bool {
            kk += by;
            bool changed = false;
            while (kk >= n_chunks && uu < end) {
                kk -= n_chunks;
                ++uu;
                changed = true;
            }
            return changed;
        };
        const long long RS = (long long)CP * A;       // sample stride of the voltages
        // slot i's row of the Re, Im (and, B tile, -Re) planes: 8 samples each
        auto put_planes = [&](unsigned char* tile, int i, const uint4& re, const uint4& im, bool neg) {
            *reinterpret_cast<uint4*>(tile + soff[i]) = re;
            *reinterpret_cast<uint4*>(tile + kPlaneBytes + soff[i]) = im;
            if (W::NEG_PLANE && neg)
                *reinterpret_cast<uint4*>(tile + 2 * kPlaneBytes + soff[i]) =
                    make_uint4(re.x ^ 0x80008000u, re.y ^ 0x80008000u, re.z ^ 0x80008000u, re.w ^ 0x80008000u);
        };
        // the same from the slot's 8 samples as (re, im) FP16 pairs x[s]
        auto put_pairs = [&](unsigned char* tile, int i, const uint32_t (&x)[8], bool neg) {
            const uint4 re = make_uint4(__byte_perm(x[0], x[1], 0x5410), __byte_perm(x[2], x[3], 0x5410),
                                        __byte_perm(x[4], x[5], 0x5410), __byte_perm(x[6], x[7], 0x5410));
            const uint4 im = make_uint4(__byte_perm(x[0], x[1], 0x7632), __byte_perm(x[2], x[3], 0x7632),
                                        __byte_perm(x[4], x[5], 0x7632), __byte_perm(x[6], x[7], 0x7632));
            put_planes(tile, i, re, im, neg);
        };
        // raw words of this thread's 8 samples (fast path: byte i = antenna 4 l + i), three chunks
        uint32_t rw0[8], rw1[8], rw2[8];
        int lu = beg, lkc = 0, lcp = 0, lab = 0, lbb = 0;                       // load cursor
        advance(lu, lkc, dset);
        if (lu < end) unit_coords(lu, nab, lcp, lab, lbb);
        const unsigned char* VB = static_cast<const unsigned char*>(a.volt);
        auto fast_load = [&](uint32_t (&w)[8]) {
#pragma unroll
            for (int s = 0; s < 8; ++s) w[s] = 0;
            if (lu < end && (bside || lab != lbb)) {
                const int col = (bside ? lbb : lab) * 128 + 4 * lane;
                if (col < A) {
                    const unsigned char* base = VB + (long long)lcp * A + col;
                    const int t0 = lkc * TC + 8 * so;
#pragma unroll
                    for (int s = 0; s < 8; ++s)
                        if (t0 + s < T) w[s] = __ldg(reinterpret_cast<const uint32_t*>(base + (long long)(t0 + s) * RS));
                }
            }
            if (advance(lu, lkc, NDS) && lu < end) unit_coords(lu, nab, lcp, lab, lbb);
        };
        // 4+4-bit words (4 samples of one slot) -> FP16 pairs: the biased nibble h = n ^ 8 in
        // [0, 15] placed under the exponent byte 0x64 is exactly 1024 + h, and 1024 + h - 1032 = n
        auto nib_pairs = [](uint32_t N, uint32_t& p01, uint32_t& p23) {
            const __half2 bias = __halves2half2(__ushort_as_half(0x6408), __ushort_as_half(0x6408));
            uint32_t u0 = __byte_perm(N, 0x64646464u, 0x4140), u1 = __byte_perm(N, 0x64646464u, 0x4342);
            const __half2 h0 = __hsub2(*reinterpret_cast<const __half2*>(&u0), bias);
            const __half2 h1 = __hsub2(*reinterpret_cast<const __half2*>(&u1), bias);
            p01 = *reinterpret_cast<const uint32_t*>(&h0);
            p23 = *reinterpret_cast<const uint32_t*>(&h1);
        };
        auto fast_decode = [&](const uint32_t (&w)[8], unsigned char* tile) {
            // rotate each sample's word so that byte i is slot i's antenna, then transpose the two
            // 4 x 4 byte blocks: q[i][h] = samples 4 h .. 4 h + 3 of slot i
            uint32_t x[8], q[4][2];
#pragma unroll
            for (int s = 0; s < 8; ++s) x[s] = __funnelshift_r(w[s], w[s], 8 * rot);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t lo01 = __byte_perm(x[4 * h], x[4 * h + 1], 0x5140);
                const uint32_t hi01 = __byte_perm(x[4 * h], x[4 * h + 1], 0x7362);
                const uint32_t lo23 = __byte_perm(x[4 * h + 2], x[4 * h + 3], 0x5140);
                const uint32_t hi23 = __byte_perm(x[4 * h + 2], x[4 * h + 3], 0x7362);
                q[0][h] = __byte_perm(lo01, lo23, 0x5410);
                q[1][h] = __byte_perm(lo01, lo23, 0x7632);
                q[2][h] = __byte_perm(hi01, hi23, 0x5410);
                q[3][h] = __byte_perm(hi01, hi23, 0x7632);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                uint4 re, im;
                // re = high nibbles, im = low nibbles, each biased by 8
                const uint32_t H0 = ((q[i][0] >> 4) & 0x0F0F0F0Fu) ^ 0x08080808u, L0 = (q[i][0] & 0x0F0F0F0Fu) ^ 0x08080808u;
                const uint32_t H1 = ((q[i][1] >> 4) & 0x0F0F0F0Fu) ^ 0x08080808u, L1 = (q[i][1] & 0x0F0F0F0Fu) ^ 0x08080808u;
                nib_pairs(H0, re.x, re.y);
                nib_pairs(H1, re.z, re.w);
                nib_pairs(L0, im.x, im.y);
                nib_pairs(L1, im.z, im.w);
                put_planes(tile, i, re, im, bside);
            }
        };
        // any voltage type, any A: slot by slot, voltage by voltage
        auto slow_decode = [&](int cp, int blk, int kc, unsigned char* tile) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int ant = blk * 128 + 4 * lane + ((i + rot) & 3);
                uint32_t x[8];
#pragma unroll
                for (int s = 0; s < 8; ++s) {
                    const int t = kc * TC + 8 * so + s;
                    const VT raw = (ant < A && t < T) ? __ldg(V + (long long)t * RS + (long long)cp * A + ant) : VT(0);
                    x[s] = voltage_pair<VDT>(raw);
                }
                put_pairs(tile, i, x, bside);
            }
        };
        if constexpr (WIDE) {
            fast_load(rw0);
            fast_load(rw1);
            fast_load(rw2);
        }
        bool failed = false;
        int cu = beg, ckc = 0, ccp = 0, cab = 0, cbb = 0;                       // decode cursor
        advance(cu, ckc, dset);
        if (cu < end) unit_coords(cu, nab, ccp, cab, cbb);
        auto one = [&](uint32_t (&rw)[8]) -> bool {
            if (cu >= end) return false;
            const int g = (cu - beg) * n_chunks + ckc;
            const int s = g % NSTAGE;
            // the stage is free once the MMAs of its previous chunk have completed
            if (g >= NSTAGE && !warp_wait(mb_empty(s), (g / NSTAGE - 1) & 1)) {
                failed = true;
                return false;
            }
            const bool diag = cab == cbb;
            unsigned char* st = sT + (size_t)s * kStageBytes;
            if (bside || !diag) {
                unsigned char* tile = bside ? st : st + kBTileBytes;
                if constexpr (WIDE) fast_decode(rw, tile);
                else slow_decode(ccp, bside ? cbb : cab, ckc, tile);
            }
            // this warp's stores, visible to the tensor cores, then its arrival
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(mb_full(s));
            // the set's third chunk from here into the registers just decoded
            if constexpr (WIDE) fast_load(rw);
            if (advance(cu, ckc, NDS) && cu < end) unit_coords(cu, nab, ccp, cab, cbb);
            return true;
        };
        // unrolled over the register sets (chosen by a branch, the sets cost 6 % of the call's time)
#pragma unroll 1
        while (one(rw0) && one(rw1) && one(rw2)) {}
        if (failed) *s_fail = 1;
    } else if (warp == MMA_WARP) {
        // ---------------- MMA warp: per K step of 16 samples two MMAs (M = 128, N = 256; or three) ----
        //   D += Re_a [Re_b; Im_b]^T,  D += Im_a [Im_b; -Re_b]^T
        // so that D[:, 0:128] = Re_a Re_b + Im_a Im_b = Re V and D[:, 128:256] = Re_a Im_b - Im_a Re_b
        // = -Im V (summed over the samples); on a diagonal unit the A planes are the B tile's.
        bool failed = false;
        int g = 0;                                // chunks whose MMAs this warp issued
        int n = 0;                                // units started
        const uint64_t d0 = sdesc(smem_u32(sT), kRowGroupBytes);
        [[maybe_unused]] constexpr uint32_t id = idesc(256), id_half = idesc(128);
        for (int u = beg; u < end && !failed; ++u, ++n) {
            int cp, ab, bb;
            unit_coords(u, nab, cp, ab, bb);
            const bool diag = ab == bb;
            const int b = n & 1;
            // accumulator buffer b is free once the epilogue has read the unit before last
            if (n >= 2 && !warp_wait(mb_acce(b), ((n >> 1) - 1) & 1)) {
                failed = true;
                break;
            }
            fence_after();
            const uint32_t tacc = tmem + 256 * b;
            for (int kc = 0; kc < n_chunks; ++kc) {
                const int s = g % NSTAGE;
                if (!warp_wait(mb_full(s), (g / NSTAGE) & 1)) {
                    failed = true;
                    break;
                }
                fence_after();
                if (lane == 0) {
                    // descriptor start fields count 16 bytes
                    const uint64_t dB1 = d0 + (uint64_t)(s * kStageBytes / 16);
                    const uint64_t dB2 = dB1 + kPlaneBytes / 16;
                    const uint64_t dA1 = diag ? dB1 : dB1 + kBTileBytes / 16;
                    const uint64_t dA2 = dA1 + kPlaneBytes / 16;
#pragma unroll
                    for (int j = 0; j < TC / 16; ++j) {
                        mma_ss(tacc, dA1 + 16 * j, dB1 + 16 * j, id, (kc | j) != 0);
                        if constexpr (W::NEG_PLANE) {
                            mma_ss(tacc, dA2 + 16 * j, dB2 + 16 * j, id, 1);
                        } else {
                            mma_ss(tacc, dA2 + 16 * j, dB2 + 16 * j, id_half, 1);
                            mma_ss(tacc + 128, dA2 + 16 * j, dB1 + 16 * j, id_half | kNegA, 1);
                        }
                    }
                    commit(mb_empty(s));
                    if (kc == n_chunks - 1) commit(mb_accf(b));
                }
                __syncwarp();
                ++g;
            }
        }
        // every MMA this warp issued has completed before the tensor memory is released
        if (g > 0) {
            if (lane == 0) commit(mb_drain);
            __syncwarp();
            mbar_wait(mb_drain, 0);
        }
        if (failed) *s_fail = 1;
    } else {
        // ---------------- epilogue warps: D -> V_ab = g_a conj(g_b) D / T (and the mirrored block) ----
        bool failed = false;
        const int q = warp & 3;                   // TMEM lane quarter this warp may read
        const float inv_t = 1.f / float(T);
        const int ew = warp - MMA_WARP - 1, c0 = ew / 4 * (512 / NEW);      // its columns: c0 .. + 512 / NEW
        float2 *rows = sRows + ew * 32 * kRowStride, *gcol = sGain + ew * 128;
        // 16-byte row stores when every row starts on a 16-byte boundary
        const bool vec = (A % 2 == 0) && ((reinterpret_cast<uintptr_t>(a.vis) & 15) == 0);
        int n = 0;
        for (int u = beg; u < end; ++u, ++n) {
            const int b = n & 1;
            int cp, ab, bb;
            unit_coords(u, nab, cp, ab, bb);
            const bool diag = ab == bb;
            const int a0 = ab * 128, b0 = bb * 128;
            const int aa = a0 + 32 * q + lane;
            const uint32_t tacc = tmem + 256 * b + ((uint32_t)(32 * q) << 16);
            // the unit's gains while its products are summed: this lane's row, and the columns in shared memory (read
            // from L2 column by column they were most of the epilogue's time)
            const float2 one = make_float2(1.f, 0.f), *gn = a.gains ? a.gains + (size_t)cp * A : nullptr;
            const float2 ga = (gn && aa < A) ? __ldg(gn + aa) : one;
#pragma unroll
            for (int i = lane; i < 128; i += 32) gcol[i] = (gn && b0 + i < A) ? __ldg(gn + b0 + i) : one;
            __syncwarp();
            if (!warp_wait(mb_accf(b), (n >> 1) & 1)) {
                failed = true;
                break;
            }
            fence_after();
            float2* out = a.vis + (size_t)cp * A * A;
            // 16 columns at a time.  A lane holds a row, so the mirrored block is written 32 adjacent elements at a
            // time, and on the diagonal, where the block is its own mirror, it alone.  Off the diagonal the rows
            // themselves go through shared memory, to be written 16 adjacent elements at a time.  Rows and columns past
            // the last antenna are left out (130 antennas: the second block column holds two).
            const int c1 = a0 + 32 * q < A ? min(c0 + 512 / NEW, A - b0) : c0;
#pragma unroll 1
            for (int c = c0; c < c1; c += 16) {
#pragma unroll
                for (int h = 0; h < 16; h += 8) {
                    float dr[8], di[8];
                    tld<8>(tacc + c + h, dr);
                    tld<8>(tacc + 128 + c + h, di);
                    tld_wait();
                    float2 v[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {                // D holds -Im V
                        const float2 gb = gcol[c + h + j];
                        const float2 w = diag ? cmul(gb, make_float2(ga.x, -ga.y)) : cmul(ga, make_float2(gb.x, -gb.y));
                        v[j] = cmul(w, make_float2(dr[j] * inv_t, (diag ? di[j] : -di[j]) * inv_t));
                        if (aa < A && b0 + c + h + j < A)
                            out[(size_t)(b0 + c + h + j) * A + aa] = make_float2(v[j].x, diag ? v[j].y : -v[j].y);
                    }
                    if (!diag) {
#pragma unroll
                        for (int j = 0; j < 8; j += 2)
                            *reinterpret_cast<float4*>(rows + lane * kRowStride + h + j) =
                                make_float4(v[j].x, v[j].y, v[j + 1].x, v[j + 1].y);
                    }
                }
                if (!diag) {
                    __syncwarp();
                    const int r0 = a0 + 32 * q;
                    if (vec && b0 + c + 16 <= A) {
#pragma unroll
                        for (int i = 0; i < 32; i += 4) {
                            const int r = i + (lane >> 3), k = 2 * (lane & 7);
                            const float4 x = *reinterpret_cast<const float4*>(rows + r * kRowStride + k);
                            if (r0 + r < A) *reinterpret_cast<float4*>(out + (size_t)(r0 + r) * A + b0 + c + k) = x;
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < 32; i += 2) {
                            const int r = i + (lane >> 4), k = lane & 15;
                            const float2 x = rows[r * kRowStride + k];
                            if (r0 + r < A && b0 + c + k < A) out[(size_t)(r0 + r) * A + b0 + c + k] = x;
                        }
                    }
                    __syncwarp();
                }
            }
            // this warp's reads of buffer b are complete: the MMA warp may overwrite it
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(mb_acce(b));
        }
        if (failed) *s_fail = 1;
    }

    fence_before();
    __syncthreads();
    if (tid == 0 && *s_fail && beg < end) {
        if (a.status) atomicOr(a.status, kStatusCorrelateTimeout);
        int cp, ab, bb;
        unit_coords(beg, nab, cp, ab, bb);
        a.vis[(size_t)cp * A * A + (size_t)(ab * 128) * A + bb * 128] =
            make_float2(__int_as_float(0x7fc00000), __int_as_float(0x7fc00000));
    }
    if (warp == MMA_WARP) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(512) : "memory");
    }
}

// ---- the FX route's imaging of an integration's visibilities (Eq. "dirty-image-FX") ----
//   U(d) = sum_{a, b} V_ab B_ab(d),  B_ab(d) = sum_g M[g, a] conj(M[g - d, b]),
//   I(k) = Re sum_d U(d) exp(+2 pi i d.k / N_p)  (image pixel order, k = 0 at the centre).
// Since B_ba(d) = conj(B_ab(-d)), the two orders of a pair add Re(S V_ab) + Re(conj(S) V_ba) to a
// pixel, S = sum_d B_ab(d) exp(+2 pi i d.k / N_p): one order with V_ab + conj(V_ba) gives the same
// image from half the table, for any visibilities (they need not be Hermitian).
// Three launches.  (1) The two orders of every pair are folded into one and written in pair-major
// order with the (channel, pol) index innermost, so that the values of one pair for consecutive
// (channel, pol) are contiguous.  (2) The lag planes are gathered from the plan's table of the antenna-pair kernels
// grouped by lag cell (B_ab(d) summed over the mapping entries of a and b once, on the host): a
// warp takes one lag cell for a group of G (channel, pol) planes, its lanes G planes x 32 / G
// entries, so that each entry's visibilities are one coalesced load for the G planes (no
// atomics; a shuffle sum over the entries).  The lag planes (wrapped mod N_p; with
// N_p >= 2 N_g - 1 none alias) go to a scratch array.  (3) One CTA per (channel, pol) takes its
// lag plane into shared memory and transforms it: N_p = S1 x S2 Cooley-Tukey per line (S2-point
// register DFTs, a twiddle, S1-point register DFTs across the line's threads), rows then
// columns, the real part written as the image.

// (1) The fold: for i < j the pair's two orders become one, W = V_ij + conj(V_ji) (or its conjugate
// where the table uses the order (j, i)); W = V_ii on the diagonal.  vis [CP][A][A] -> vis_t
// [pair][CP], pair = the packed index of i <= j.  A block takes FXT_A rows i and 32 columns j for 32
// planes: V_ij is read 32 columns (256 bytes) at a time, V_ji 4 columns (one 32-byte sector) of 32
// rows, and 32 planes of a pair are written as 256 bytes.  HBM-bound: every visibility is read once.
constexpr int FXT_A = 4;
constexpr int FXT_J = 33, FXT_I = 32 * FXT_J + 4;   // strides of the tile (float2): no bank conflicts

__global__ void __launch_bounds__(256) fx_fold_kernel(const float2* __restrict__ vis, int n_cp, int A,
                                                      float2* __restrict__ vis_t) {
    __shared__ float2 tile[FXT_A * FXT_I];
    const int j0 = blockIdx.x * 32, i0 = blockIdx.y * FXT_A, c0 = blockIdx.z * 32;
    if (j0 + 31 < i0) return;                       // below the diagonal
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const size_t plane = (size_t)A * A;
    // V_ij: a warp reads the 32 columns of one (row, plane)
#pragma unroll 4
    for (int q = warp; q < FXT_A * 32; q += 8) {
        const int i = i0 + q / 32, c = c0 + q % 32, j = j0 + lane;
        if (c < n_cp && i < A && j < A && j >= i)
            tile[(q / 32) * FXT_I + lane * FXT_J + q % 32] = __ldg(vis + (size_t)c * plane + (size_t)i * A + j);
    }
    __syncthreads();
    // V_ji: 4 columns i of 8 rows j
#pragma unroll 4
    for (int q = warp; q < 4 * 32; q += 8) {
        const int ii = lane & 3, jj = (q / 32) * 8 + (lane >> 2), cc = q % 32;
        const int i = i0 + ii, j = j0 + jj, c = c0 + cc;
        if (c < n_cp && j < A && j > i) {
            const float2 u = __ldg(vis + (size_t)c * plane + (size_t)j * A + i);
            float2* t = tile + ii * FXT_I + jj * FXT_J + cc;
            const float2 v = make_float2(t->x + u.x, t->y - u.y);
            *t = fx_pair_swapped(i, j) ? make_float2(v.x, -v.y) : v;
        }
    }
    __syncthreads();
    for (int q = warp; q < FXT_A * 32; q += 8) {
        const int i = i0 + q / 32, j = j0 + q % 32, c = c0 + lane;
        if (c < n_cp && i < A && j < A && j >= i) {
            const size_t pair = (size_t)i * A - (size_t)i * (i - 1) / 2 + (j - i);
            vis_t[pair * n_cp + c] = tile[(q / 32) * FXT_I + (q % 32) * FXT_J + lane];
        }
    }
}

// (2) U[cp][d] = sum over the entries of lag cell d of vis_t[off / CP][cp] * B (each entry
// holds the element offset off = pair * CP of its pair's row).  A CTA takes an 8 x 8 tile of lag
// cells (neighbouring cells share most of their pairs, which then stay in L1) for one group of
// G planes; the CTAs of one tile (all groups) are adjacent in launch order so that they share
// the tile's table entries in L2.  A warp takes whole lag cells.  It reads the entries of a cell
// 32 at a time with one coalesced load into its own shared-memory slots (slots past the cell's
// end hold zero weights at offset 0; the next 32 entries are loaded while these are used).  An
// entry takes G / W lanes of W planes each, E = 32 W / G entries side by side, and the sum over a
// cell's entries ends with a shuffle.  V4 (an even number of planes): W = 2, one 16-byte load per
// lane and entry; else W = 1 with 8-byte loads.
//
// What bounds it: the visibilities' way from L2 to L1 (each pair is used by up to 81 lag cells), then
// L1 wavefronts, and for few planes the tiles around lag 0, which hold several times the mean number
// of entries.  Measured on a 256-antenna layout (N_p = 128; all three launches): 965 us at 128 planes
// with both orders of every pair gathered, G = 64 and 8-warp CTAs; 538 with one order; 412 with
// G = 16 (a tile's pairs then mostly stay in L1); 286 with the tiles ordered by their distance from
// lag 0; 229 with one 32-warp CTA per SM, which shortens the longest tiles fourfold (64 registers,
// 4 loads in flight per lane).  The width G: see fx_planes_per_group.
constexpr int FXG_NT = 1024;

template <int G, bool V4>
__global__ void __launch_bounds__(FXG_NT, 1) fx_gather_kernel(const FxArgs a, int np) {
    static_assert(G <= 32 && (!V4 || G >= 2), "group width");
    constexpr int W = V4 ? 2 : 1;                                        // planes per lane
    constexpr int LPE = G / W;                                           // lanes per entry
    constexpr int E = 32 / LPE;                                          // entry slots per step
    constexpr int U0 = V4 ? 4 : 16;
    constexpr int U = (U0 * E <= 32) ? U0 : 32 / E;                      // entries per lane in flight
    static_assert(U * E <= 32 && 32 % (U * E) == 0, "steps");
    __shared__ int4 sent[FXG_NT / 32][32];
    const int CP = a.n_cp, n_groups = (CP + G - 1) / G;
    const int tiles_x = np / 8;
    const int tile = blockIdx.x / n_groups, gi = blockIdx.x - tile * n_groups;
    // tiles in the order of their distance from lag 0 (the wrapped corners), where most pairs lie, so
    // that the longest blocks start first: the tile number's even and odd bits are the positions
    // along x and y, position p the p-th nearest tile row to lag 0
    int ix = 0, iy = 0;
    for (int bit = 0; (1 << bit) < tiles_x; ++bit) {
        ix |= ((tile >> (2 * bit)) & 1) << bit;
        iy |= ((tile >> (2 * bit + 1)) & 1) << bit;
    }
    const int ty0 = 8 * ((iy & 1) ? tiles_x - 1 - iy / 2 : iy / 2), tx0 = 8 * ((ix & 1) ? tiles_x - 1 - ix / 2 : ix / 2);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int e = lane / LPE;
    const int cp = gi * G + W * (lane % LPE);                            // first plane of the lane
    const bool valid = cp < CP;                                          // (V4: CP is even)
    const float2* Vt = a.vis_t + (valid ? cp : 0);
    int4* sw = sent[warp];
    for (int j = warp; j < 64; j += FXG_NT / 32) {
        const int d = (ty0 + (j >> 3)) * np + tx0 + (j & 7);
        const int p0 = __ldg(a.lag_ptr + d), p1 = __ldg(a.lag_ptr + d + 1);
        float2 acc[W] = {};
        int4 nxt = p0 + lane < p1 ? __ldg(a.lag_ent + p0 + lane) : make_int4(0, 0, 0, 0);
        for (int q0 = p0; q0 < p1; q0 += 32) {
            const int nb = min(32, p1 - q0);
            __syncwarp();
            sw[lane] = nxt;
            __syncwarp();
            nxt = q0 + 32 + lane < p1 ? __ldg(a.lag_ent + q0 + 32 + lane) : make_int4(0, 0, 0, 0);
            for (int k = 0; k < nb; k += U * E) {
                float2 v[U][W], w[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int4 en = sw[k + u * E + e];
                    w[u] = make_float2(__int_as_float(en.x), __int_as_float(en.y));
                    if constexpr (V4) {
                        const float4 f = __ldg(reinterpret_cast<const float4*>(Vt + en.z));
                        v[u][0] = make_float2(f.x, f.y);
                        v[u][1] = make_float2(f.z, f.w);
                    } else {
                        v[u][0] = __ldg(Vt + en.z);
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int i = 0; i < W; ++i) {
                        acc[i].x = fmaf(v[u][i].x, w[u].x, fmaf(-v[u][i].y, w[u].y, acc[i].x));
                        acc[i].y = fmaf(v[u][i].x, w[u].y, fmaf(v[u][i].y, w[u].x, acc[i].y));
                    }
            }
        }
        const size_t npix = (size_t)np * np;
#pragma unroll
        for (int i = 0; i < W; ++i) {
#pragma unroll
            for (int o = 16; o >= LPE; o >>= 1) {
                acc[i].x += __shfl_xor_sync(0xffffffffu, acc[i].x, o);
                acc[i].y += __shfl_xor_sync(0xffffffffu, acc[i].y, o);
            }
            if (e == 0 && valid) a.u[(size_t)(cp + i) * npix + d] = acc[i];
        }
    }
}

// (3) the transform of one lag plane.  Line of length NP = S1 x S2, n = S1 m + r, k = k1 + S2 k2:
//   X[k1 + S2 k2] = sum_r exp(2 pi i r k2 / S1) [exp(2 pi i r k1 / NP) Y_r[k1]],
//   Y_r[k1] = sum_m x[S1 m + r] exp(2 pi i m k1 / S2).
// Thread (line, r) computes Y_r in registers and stores Y_r[k1] at line position
// r S2 + (k1 xor r) (the xor spreads the S1 threads of a line over distinct banks); thread
// (line, r') then takes k1 = r' + S1 i and does the S1-point DFTs.  Rows are padded to NP + S1
// elements so that the lines a warp touches fall into complementary halves of the banks.  The
// centring (k measured from N_p / 2) is the sign (-1)^(dx + dy) applied to U on loading.
template <int NP>
struct FxDft {
    static constexpr int S1 = NP == 32 ? 4 : 8, S2 = NP / S1, NT = 4 * NP, P = NP + S1;
    static constexpr size_t smem = sizeof(float2) * ((size_t)NP * P + NP);
};

template <int NP>
__global__ void __launch_bounds__(FxDft<NP>::NT) fx_dft_kernel(const float2* __restrict__ u, float* __restrict__ image) {
    using D = FxDft<NP>;
    constexpr int S1 = D::S1, S2 = D::S2, NT = D::NT, P = D::P, MSK = NP - 1;
    static_assert(S1 * S2 == NP && S2 >= S1 && NT % NP == 0, "factorisation");
    extern __shared__ __align__(16) unsigned char fx_smem[];
    float2* L = reinterpret_cast<float2*>(fx_smem);       // [NP][P]
    float2* TW = L + NP * P;                               // [NP] exp(+2 pi i j / NP)
    const int tid = threadIdx.x, cp = blockIdx.x;
    for (int j = tid; j < NP; j += NT) {
        double s, c;
        sincospi(2.0 * j / NP, &s, &c);
        TW[j] = make_float2(float(c), float(s));
    }
    const float2* U = u + (size_t)cp * NP * NP;
    for (int i = tid; i < NP * NP; i += NT) {
        const int dy = i / NP, dx = i % NP;
        float2 v = __ldg(U + i);
        if ((dx + dy) & 1) v = make_float2(-v.x, -v.y);
        L[dy * P + dx] = v;
    }
    __syncthreads();
    // rows: line dy, element dx at L[dy * P + dx]
    {
        constexpr int LPI = NT / S1;                        // lines per iteration
        const int r = tid % S1;
#pragma unroll 1
        for (int l0 = 0; l0 < NP; l0 += LPI) {
            float2* row = L + (l0 + tid / S1) * P;
            float2 x[S2];
#pragma unroll
            for (int m = 0; m < S2; ++m) x[m] = row[S1 * m + r];
            dft<S2, 1>(x);
#pragma unroll
            for (int k1 = 1; k1 < S2; ++k1) x[k1] = cmul(x[k1], TW[(r * k1) & MSK]);
            __syncthreads();
#pragma unroll
            for (int k1 = 0; k1 < S2; ++k1) row[r * S2 + (k1 ^ r)] = x[k1];
        }
        __syncthreads();
#pragma unroll 1
        for (int l0 = 0; l0 < NP; l0 += LPI) {
            float2* row = L + (l0 + tid / S1) * P;
            float2 y[S2 / S1][S1];
#pragma unroll
            for (int i = 0; i < S2 / S1; ++i) {
                const int k1 = r + S1 * i;
#pragma unroll
                for (int q = 0; q < S1; ++q) y[i][q] = row[q * S2 + (k1 ^ q)];
                dft<S1, 1>(y[i]);
            }
            __syncthreads();
#pragma unroll
            for (int i = 0; i < S2 / S1; ++i)
#pragma unroll
                for (int k2 = 0; k2 < S1; ++k2) row[r + S1 * i + S2 * k2] = y[i][k2];
        }
    }
    __syncthreads();
    // columns: line ix, element dy at L[dy * P + ix]; thread -> (ix = tid % NP, r), a warp 32
    // consecutive columns
    {
        constexpr int RPI = NT / NP, RIT = S1 / RPI;        // r values per iteration, iterations
        static_assert(RPI * RIT == S1, "column split");
        const int ix = tid % NP;
        // every r of a column is read before any is overwritten (the iterations share columns)
        float2 x[RIT][S2];
#pragma unroll
        for (int it = 0; it < RIT; ++it) {
            const int r = RPI * it + tid / NP;
#pragma unroll
            for (int m = 0; m < S2; ++m) x[it][m] = L[(S1 * m + r) * P + ix];
            dft<S2, 1>(x[it]);
#pragma unroll
            for (int k1 = 1; k1 < S2; ++k1) x[it][k1] = cmul(x[it][k1], TW[(r * k1) & MSK]);
        }
        __syncthreads();
#pragma unroll
        for (int it = 0; it < RIT; ++it) {
            const int r = RPI * it + tid / NP;
#pragma unroll
            for (int k1 = 0; k1 < S2; ++k1) L[(r * S2 + (k1 ^ r)) * P + ix] = x[it][k1];
        }
        __syncthreads();
        float* img = image + (size_t)cp * NP * NP;
#pragma unroll 1
        for (int r0 = 0; r0 < S1; r0 += RPI) {
            const int r = r0 + tid / NP;
#pragma unroll
            for (int i = 0; i < S2 / S1; ++i) {
                const int k1 = r + S1 * i;
                float2 y[S1];
#pragma unroll
                for (int q = 0; q < S1; ++q) y[q] = L[(q * S2 + (k1 ^ q)) * P + ix];
                dft<S1, 1>(y);
#pragma unroll
                for (int k2 = 0; k2 < S1; ++k2) img[(size_t)(k1 + S2 * k2) * NP + ix] = y[k2].x;
            }
        }
    }
}

template <int NP>
cudaError_t launch_fx_image_t(const FxArgs& a, cudaStream_t st) {
    fx_fold_kernel<<<dim3((unsigned)((a.n_ant + 31) / 32), (unsigned)((a.n_ant + FXT_A - 1) / FXT_A),
                          (unsigned)((a.n_cp + 31) / 32)), 256, 0, st>>>(a.vis, a.n_cp, a.n_ant, a.vis_t);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int g = fx_planes_per_group(a.n_cp, NP, a.n_ent);
    const unsigned blocks = (unsigned)((NP / 8) * (NP / 8) * (long long)((a.n_cp + g - 1) / g));
    switch (2 * g + (a.n_cp % 2 == 0 ? 1 : 0)) {
        case 2: fx_gather_kernel<1, false><<<blocks, FXG_NT, 0, st>>>(a, NP); break;
        case 4: fx_gather_kernel<2, false><<<blocks, FXG_NT, 0, st>>>(a, NP); break;
        case 5: fx_gather_kernel<2, true><<<blocks, FXG_NT, 0, st>>>(a, NP); break;
        case 8: fx_gather_kernel<4, false><<<blocks, FXG_NT, 0, st>>>(a, NP); break;
        case 9: fx_gather_kernel<4, true><<<blocks, FXG_NT, 0, st>>>(a, NP); break;
        case 16: fx_gather_kernel<8, false><<<blocks, FXG_NT, 0, st>>>(a, NP); break;
        case 17: fx_gather_kernel<8, true><<<blocks, FXG_NT, 0, st>>>(a, NP); break;
        case 32: fx_gather_kernel<16, false><<<blocks, FXG_NT, 0, st>>>(a, NP); break;
        case 33: fx_gather_kernel<16, true><<<blocks, FXG_NT, 0, st>>>(a, NP); break;
        case 64: fx_gather_kernel<32, false><<<blocks, FXG_NT, 0, st>>>(a, NP); break;
        default: fx_gather_kernel<32, true><<<blocks, FXG_NT, 0, st>>>(a, NP); break;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    using D = FxDft<NP>;
    if ((e = ensure_smem<fx_dft_kernel<NP>>(D::smem)) != cudaSuccess) return e;
    fx_dft_kernel<NP><<<a.n_cp, D::NT, D::smem, st>>>(a.u, a.image);
    return cudaGetLastError();
}

}  // namespace xe

size_t xeng_smem_bytes() {
    return std::max({xe::Roles<false, false>::kSmem, xe::Roles<false, true>::kSmem, xe::Roles<true, false>::kSmem});
}

cudaError_t launch_fx_image(int n_pad, const FxArgs& a, cudaStream_t st) {
    if (a.n_cp == 0) return cudaSuccess;
    switch (n_pad) {
        case 32: return xe::launch_fx_image_t<32>(a, st);
        case 64: return xe::launch_fx_image_t<64>(a, st);
        case 128: return xe::launch_fx_image_t<128>(a, st);
        default: return cudaErrorInvalidValue;
    }
}

namespace {
template <int VDT, bool WIDE, bool SHORT>
cudaError_t launch_xeng_t(const XengArgs& a, long long grid, cudaStream_t st) {
    constexpr size_t smem = xe::Roles<WIDE, SHORT>::kSmem;
    const cudaError_t e = ensure_smem<xe::xeng_kernel<VDT, WIDE, SHORT>>(smem);
    if (e != cudaSuccess) return e;
    xe::xeng_kernel<VDT, WIDE, SHORT><<<(unsigned)grid, xe::Roles<WIDE, SHORT>::NT, smem, st>>>(a);
    return cudaGetLastError();
}

template <int VDT>
cudaError_t launch_xeng_singly(const XengArgs& a, long long grid, cudaStream_t st) {
    return xeng_short(VDT == 1, a.n_time) ? launch_xeng_t<VDT, false, true>(a, grid, st)
                                          : launch_xeng_t<VDT, false, false>(a, grid, st);
}
}  // namespace

cudaError_t launch_xeng(int vdt, const XengArgs& a, int n_sm, cudaStream_t st) {
    const int nab = (a.n_ant + 127) / 128;
    const long long n_units = (long long)a.n_cp * (nab * (nab + 1) / 2);
    if (n_units == 0) return cudaSuccess;
    if (n_units > 2147483647LL) return cudaErrorInvalidValue;   // the kernel indexes units in 32 bits
    const long long grid = n_units < n_sm ? n_units : n_sm;
    switch (vdt) {
        case 1:
            return launch_xeng_singly<1>(a, grid, st);
        case 2:
            // 4-byte loads of 4 antennas need every group of 4 to start on a 4-byte boundary
            if (a.n_ant % 4 == 0 && reinterpret_cast<uintptr_t>(a.volt) % 4 == 0)
                return launch_xeng_t<2, true, false>(a, grid, st);
            return launch_xeng_singly<2>(a, grid, st);
        default:
            return cudaErrorInvalidValue;
    }
}

}  // namespace epic
