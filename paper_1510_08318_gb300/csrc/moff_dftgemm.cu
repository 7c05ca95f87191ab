// MOFF imaging with the spatial transform as a dense DFT on the 5th-generation tensor cores
// (Eq. "dirty-image-MOFF"; the transform of Sec. 3 "Spatial Fourier Transform" written as two
// matrix products), N_p = 128 (N_g = 64):
//
//   X(ky, x)  = sum_y  W[ky][y] E(y, x)          stage 1
//   F(ky, kx) = sum_x  X(ky, x) W[kx][x]         stage 2
//   I(ky, kx) += |F|^2
//
// with W[k][n] = exp(+2 pi i n k / N_p).  The frequencies are taken in pairs.  The gridded field is
// multiplied by exp(-i pi (x + y) / N_p), which moves the frequencies by a half: k becomes k + 1/2,
// and k = 0 .. 63 and -1 .. -64 are 64 pairs +-(k + 1/2).  With C[k][n] = cos(2 pi n (k + 1/2) / N_p)
// and S[k][n] the sine, one product with the 128 rows [C ; S] gives P = C E and Q = S E, and both
// frequencies of a pair follow by additions, P + i Q and P - i Q: half the products of the dense form,
// in both stages, and half the table.
//
// Every real operand v is split as v = hi + lo (two FP16 numbers, hi = fp16(v), lo = fp16(v - hi))
// and each real product is hi*hi + hi*lo + lo*hi accumulated in FP32 in tensor memory (about 22 bits
// of operand precision).  Per image the gridded field is scaled by a power of two, chosen from a
// bound (largest |g V| of the sample times the largest sum_a |M[g, a]| of the plan), so that the
// FP16 operands stay in range; |F|^2 is scaled back exactly.
//
// Two consecutive images A and B are processed together: a mapping entry read by the gridding serves
// both (their voltages are one 16-byte word per antenna).
// Table rows (and tensor-memory lanes) are ordered C 0..15, S 0..15, C 16..31, S 16..31, ...
//   Stage 1: A operand = the table (M = 128), B operand = the rows [Re A, Im A, Re B, Im B] of E^T
//     (N = 128 each, K = 64): 12 MMAs per image.  In each warp's 32 lanes the first 16 then hold P, the
//     other 16 hold Q of the same k.
//   Split, image by image: a lane takes the value v of the lane 16 away and forms own + i v, which is
//     X(k) = P + i Q in the P lanes and Q + i P = i (P - i Q) = i X(-k - 1) in the Q lanes (the factor i of
//     a whole image row leaves |F|^2 as it is), 16 x per thread, and writes it back as FP16 hi and lo
//     into the columns it read.
//   Stage 2 of an image: A operand from tensor memory (its lanes are the image's 128 ky) against the
//     table as B operand (N = 128): F = re (128 columns), im (128 columns), 24 MMAs.
//   Epilogue: a thread's columns C, S of re and im give F(ky, kx) and F(ky, -kx - 1) by additions.
//
// One CTA per SM: 16 transform warps (split, epilogue), 11 gridding warps (decode, gridding) and one warp
// whose first thread issues the MMAs.  It owns all 512 TMEM columns:
//   [0, 256)    stage-1 accumulator (A, then B), then the stage-2 A operands in the same columns
//   [256, 512)  F of one image
// Shared memory: the table (hi, lo; 32 KB), two buffers of the E^T operand (64 KB each), the voltages of
// two pairs of images (of one where two do not fit), per-antenna powers, and the gather tables where they
// fit beside these.
//
// The roles meet at mbarriers only.  Gridding warps, per pair p: decode it, and once all of them have, grid
// it into E buffer p mod 2 (free after stage 1 of pair p - 2).  Issuer, image by image: stage 2 of image i
// (split, and F of image i - 1 taken), and once it is done stage 1 of image i + 2, whose accumulator takes
// the columns of image i's operand.  Transform warps: split image i + 1, take F of image i.  So stage 2 of
// an image runs beside the split of the next one, and stage 1 beside the taking of F.
//
// Why this form.  Measured on 256 antennas, 4+4-bit, 262,144 images (ms a call): 6.89 with the dense
// products (72 MMAs an image), one image at a time, one gather entry per mapping entry and every warp
// doing every step: 20,900 warp instructions an image at 67 % of the issue slots.  5.88 with frequency
// pairs and two images per gather entry (16,000 instructions).  Stage 2 in two parts of N = 64, to take F
// of one while the other runs, was slower than N = 128: an N = 64 MMA takes as long (8,200 cycles a pair
// for the MMAs alone, 6,500 with N = 128, 4,600 at the nominal rate).  5.56 with entries of equal steps
// (no per-lane counts).  The exchange of P and Q through shared memory took 5,900 cycles a pair, the
// shuffles a third of it.  5.12 with each part once in the code (unrolled into every place of use, the loop
// ran out of the instruction cache).  3.96 with gridding and transform warps apart (13,500 -> 11,000
// instructions, and their latencies side by side), 3.66 with the images one behind the other in the
// tensor pipe instead of pair after pair.  Now: the gridding warps alone take 80 % of it, the MMAs alone 70 %.
//
// The gridding gathers cell pairs (x, y), (x, y + 1) from slot tables in which the 32 pairs of a warp
// step have similar entry counts and store to 32 distinct shared-memory banks.  An entry is an antenna
// with its weights on both cells (0 where it has none): on the 256-antenna ellipse 4,079
// entries for 6,707 mapping entries, 159 warp steps of two images where the cells' own entries took 258
// of one.  The builder orders a pair's entries so that the antennas read at one warp
// step spread over the shared-memory banks of the 16-byte voltages (a fixed order: the sums are
// deterministic).
// Every wait is bounded (by the plan's try count) and taken by a whole warp; on a timeout the role
// stops, the CTA sets the image-timeout bit of the plan's status word, writes NaN into its
// accumulator block, and the issuer waits with the full limit for the MMAs it issued before the
// tensor memory is released.
#include <cuda_fp16.h>
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <type_traits>
#include <vector>
#include "moff_common.cuh"
#include "tcgen05.cuh"

namespace epic {
namespace dg {
using namespace tc;

constexpr int NP = 128, NG = 64;
constexpr int NXW = 16;                   // transform warps: 4 per TMEM lane quarter
constexpr int NGW = 11;                   // gridding warps
constexpr int NTH = 32 * (NXW + NGW + 1); // + the issuer's warp
constexpr int NGT = 32 * NGW;             // gridding threads
// Registers: 896 threads are launched with at most 72 each, shared out by whole groups of four warps: the transform warps
// (32 FP32 sums and 32 columns in flight) take 88 and the others 48, or 80 and 56 in the forms whose gridding warps need
// more (two voltages a decode for XP) or whose transform warps need less (LP).  Measured (us): 262,144 images 3,675 and
// 3,718; XP 32,768 images 565 and 549; LP 262,144 images 3,328 and 3,287.
constexpr int regs_transform(bool xp, bool lp) { return xp || lp ? 80 : 88; }
constexpr int regs_other(bool xp, bool lp) { return xp || lp ? 56 : 48; }
constexpr bool split_fits(bool xp, bool lp) {
    return NXW * regs_transform(xp, lp) + (NGW + 1) * regs_other(xp, lp) <= (NXW + NGW + 1) * 72;
}
static_assert((NXW % 4) == 0 && ((NGW + 1) % 4) == 0 && split_fits(false, false) && split_fits(true, false) &&
                  split_fits(false, true), "register split");
constexpr int WTAB = NP * NG;     // halves per [C ; S] table (hi or lo)
constexpr int EIMG = 2 * NG * NG; // halves of one image's [Re ; Im] E^T rows
constexpr int EPART = 2 * EIMG;   // halves of a pair's hi (or lo) E^T rows
constexpr int ebuf(bool lp) { return (lp ? 1 : 2) * EPART; }   // halves per E buffer: hi, lo (LP: hi)
constexpr int NSLOT = NG * NG / 64;   // slots of 32 cell pairs
constexpr int PER_WARP = (NSLOT + NGW - 1) / NGW, NPOS = NGW * PER_WARP;   // slot positions of the gridding warps
// mbarriers.  E full and E free have one per parity of the pair (the gridding may be two pairs ahead), stage
// 1 done one per image of a pair.
enum { MB_EFULL, MB_VFULL = MB_EFULL + 2, MB_XA, MB_XB, MB_FREE, MB_ST1, MB_EFREE = MB_ST1 + 2, MB_F = MB_EFREE + 2, MB_DRAIN,
       N_MBAR };

// packed FP32 pair (a, b) -> FP16 pairs hi = fp16(a, b), lo = fp16((a, b) - hi)
__device__ __forceinline__ void split2(unsigned long long ab, uint32_t& hi, uint32_t& lo) {
    const float2 v = unpack2(ab);
    const __half2 h = __floats2half2_rn(v.x, v.y);
    const float2 d = unpack2(f2sub(ab, pack2(__half22float2(h))));
    const __half2 l = __floats2half2_rn(d.x, d.y);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}
__device__ __forceinline__ uint32_t half_pair(unsigned long long ab) {
    const float2 v = unpack2(ab);
    const __half2 h = __floats2half2_rn(v.x, v.y);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// Shared memory before the per-antenna arrays: the table (the reduced-precision form LP keeps the hi
// parts only), two E buffers, the mbarriers and small words.
constexpr size_t kMiscBytes = 256;
constexpr size_t smem_fixed(bool lp = false) {
    return sizeof(__half) * ((size_t)(lp ? 1 : 2) * WTAB + 2 * (size_t)ebuf(lp)) + kMiscBytes;
}
static_assert(8 * N_MBAR + 2 * 4 + 32 * 4 <= kMiscBytes, "mbarriers and words");
// Shared-memory bytes per antenna: nvb buffers of a pair's voltages (2 float2, or 2 half2 in the LP
// form) and the power.
constexpr size_t ant_bytes(bool lp, int nvb) { return (size_t)nvb * (lp ? 8 : 16) + 4; }

// FP16 rounding of a float (the reduced-precision form's operands)
__device__ __forceinline__ float round_h(float x) { return __half2float(__float2half_rn(x)); }

// Bytes of the gather tables when they are copied into shared memory (after the per-antenna
// arrays, 16-byte aligned): weights (and imaginary parts), slots, antennas.
inline size_t table_smem_bytes(int n_ent, bool cw) {
    return 16 + sizeof(float2) * (size_t)n_ent * (cw ? 2 : 1) + sizeof(int2) * NPOS + sizeof(uint16_t) * (size_t)n_ent;
}

// Gather-table load: shared memory when the tables were copied there, else the read-only path.
template <bool SMT, typename T>
__device__ __forceinline__ T ldt(const T* p) {
    if constexpr (SMT) return *p;
    else return __ldg(p);
}

template <int VDT, bool SMT, bool XP, bool LP>
__global__ void __launch_bounds__(NTH, 1) moff_dftgemm_kernel(const FwdArgs a, const __half* __restrict__ wtab,
                                                              const DgPairGather g, const int nvb) {
    using VT = typename Volt<VDT>::T;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    constexpr int NWT = LP ? 1 : 2, EBUF = ebuf(LP);
    constexpr int kRegsTransform = regs_transform(XP, LP), kRegsOther = regs_other(XP, LP);
    __half* sW = reinterpret_cast<__half*>(smem_raw);                      // [NWT][WTAB]
    __half* sE = sW + NWT * WTAB;                                         // [2][EBUF]
    uint64_t* mbar = reinterpret_cast<uint64_t*>(sE + 2 * EBUF);          // [N_MBAR]
    uint32_t* tslot = reinterpret_cast<uint32_t*>(mbar + N_MBAR);
    int* s_fail = reinterpret_cast<int*>(tslot + 1);
    unsigned int* vmax = reinterpret_cast<unsigned int*>(tslot + 2);      // [16][2] max |g V| (float bits) per pair mod 16
    const int A = a.n_ant, T = a.n_time;
    unsigned char* sVB = smem_raw + smem_fixed(LP);                       // [nvb][A] a pair's voltages
    constexpr int VBYTES = LP ? 8 : 16;
    float* PW = reinterpret_cast<float*>(sVB + (size_t)nvb * A * VBYTES);
    float2* sWre = reinterpret_cast<float2*>(smem_raw + ((smem_fixed(LP) + (size_t)A * ant_bytes(LP, nvb) + 15) & ~(size_t)15));
    float2* sWim = sWre + g.n_ent;
    int2* sSlot = reinterpret_cast<int2*>(sWre + (g.wim ? 2 : 1) * g.n_ent);
    uint16_t* sAnt = reinterpret_cast<uint16_t*>(sSlot + NPOS);
    const float2* tWre = SMT ? sWre : g.w;
    const float2* tWim = g.wim == nullptr ? nullptr : SMT ? sWim : g.wim;
    const int2* tSlot = SMT ? sSlot : g.slot;
    const uint16_t* tAnt = SMT ? sAnt : g.ant;
    const float4* rot = reinterpret_cast<const float4*>(wtab + 2 * WTAB);   // cos and sin of pi s / NP, s and s + 1

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const VT* V = static_cast<const VT*>(a.volt);
    auto mb = [&](int i) { return smem_u32(&mbar[i]); };
    // a bounded wait taken by a whole warp: the warp goes on only if every lane saw the phase
    auto warp_wait = [&](int i, int parity) -> bool {
        return __all_sync(0xffffffffu, mbar_wait(mb(i), (uint32_t)parity & 1u, a.wait_tries)) != 0;
    };
    // one arrival per warp, after everything its lanes did before
    auto warp_arrive = [&](int i) {
        __syncwarp();
        if (lane == 0) mbar_arrive(mb(i));
    };

    for (int i = tid; i < NWT * WTAB / 8; i += NTH)
        reinterpret_cast<uint4*>(sW)[i] = __ldg(reinterpret_cast<const uint4*>(wtab) + i);
    for (int aa = tid; aa < A; aa += NTH) PW[aa] = 0.f;
    if constexpr (SMT) {
        for (int q = tid; q < NPOS; q += NTH) sSlot[q] = __ldg(g.slot + q);
        for (int q = tid; q < g.n_ent; q += NTH) {
            sWre[q] = __ldg(g.w + q);
            sAnt[q] = __ldg(g.ant + q);
        }
        if (g.wim)
            for (int q = tid; q < g.n_ent; q += NTH) sWim[q] = __ldg(g.wim + q);
    }
    if (tid == 0) {
        for (int i = 0; i < N_MBAR; ++i)
            mbar_init(mb(i), i <= MB_VFULL ? NGW : i <= MB_FREE ? NXW : 1);
        *s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(tslot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid < 32) vmax[tid] = 0u;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");          // the table, for the tensor cores
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tslot;
    const uint32_t tX = tmem, tF = tmem + 256;

    long long beg_l, end_l;
    work_range(a.n_items, blockIdx.x, gridDim.x, beg_l, end_l);
    const int beg = (int)beg_l, n = (int)(end_l - beg_l);
    const int np = (n + 1) / 2;               // pairs of images; the last one may hold one image

    auto exponent = [&](int p, int img) -> int {
        // |E| <= (largest sum_a |M[g, a]|) * sqrt(2) * (largest |g V| component)
        const float bound = a.wsum_max * 1.5f * __uint_as_float(vmax[2 * (p & 15) + img]);
        const int ex = (int)(__float_as_uint(bound) >> 23) - 126 - 9;     // scaled bound in [256, 512)
        return bound > 0.f ? max(-100, min(100, ex)) : 0;
    };

    if (warp < NXW) {
        // ------------------------------- transform warps -------------------------------
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" :: "n"(kRegsTransform));
        const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
        const int qt = warp >> 2;                       // the 16 x of its split, the 16 kx of its epilogue
        const int kk = 16 * (warp & 3) + (lane & 15);   // its ky: row kk (lanes 0..15), or -(kk + 1)

        unsigned long long acc[2][8];                   // [plus, minus kx][pairs of kx]
#pragma unroll
        for (int i = 0; i < 16; ++i) (&acc[0][0])[i] = 0ull;

        // ---- split of image img (after its stage 1) ----
        // This warp's columns: 16 re (block 0) and 16 im (block 1, 64 columns on).  They become the A operand:
        // re hi and im hi in block 0 (8 columns each), re lo and im lo in block 1.
        auto split = [&](int img) {
            const uint32_t own = tX + lane_base + 128 * img + 16 * qt;
            float vr[16], vi[16];
            tld<16>(own, vr);
            tld<16>(own + 64, vi);
            tld_wait();
            uint32_t rh[8], rl[8], ih[8], il[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                float2 xr, xi, br, bi;
                br = make_float2(__shfl_xor_sync(0xffffffffu, vr[2 * u], 16), __shfl_xor_sync(0xffffffffu, vr[2 * u + 1], 16));
                bi = make_float2(__shfl_xor_sync(0xffffffffu, vi[2 * u], 16), __shfl_xor_sync(0xffffffffu, vi[2 * u + 1], 16));
                xr = make_float2(vr[2 * u], vr[2 * u + 1]);
                xi = make_float2(vi[2 * u], vi[2 * u + 1]);
                const unsigned long long sr = f2sub(pack2(xr), pack2(bi)), si = f2add(pack2(xi), pack2(br));
                if constexpr (LP) {
                    rh[u] = half_pair(sr);
                    ih[u] = half_pair(si);
                } else {
                    split2(sr, rh[u], rl[u]);
                    split2(si, ih[u], il[u]);
                }
            }
            tst8(own, rh);
            tst8(own + 8, ih);
            if constexpr (!LP) {
                tst8(own + 64, rl);
                tst8(own + 72, il);
            }
            tst_wait();
            fence_before();
            warp_arrive(MB_XA + img);
        };

        // ---- epilogue ----
        // F of image img: re and im of 128 columns each, blocks of 16 C and 16 S; this thread's 16 kx
        auto epilogue = [&](int p, int img) -> bool {
            const unsigned long long sc2 = f2dup(ldexpf(1.f, 2 * exponent(p, img)));
            if (!warp_wait(MB_F, img)) return false;
            fence_after();
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float v[4][8];                              // C re, S re, C im, S im of 8 kx
#pragma unroll
                for (int c = 0; c < 4; ++c) tld<8>(tF + 128 * (c >> 1) + lane_base + 32 * qt + 16 * (c & 1) + 8 * h, v[c]);
                tld_wait();
                if (h == 1) {                               // F may be overwritten
                    fence_before();
                    warp_arrive(MB_FREE);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    unsigned long long d[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) d[c] = pack2(make_float2(v[c][2 * u], v[c][2 * u + 1]));
                    // F(kx) = C + i S, F(-kx - 1) = C - i S
                    const unsigned long long pr = f2sub(d[0], d[3]), pi = f2add(d[2], d[1]);
                    const unsigned long long mr = f2add(d[0], d[3]), mi = f2sub(d[2], d[1]);
                    acc[0][4 * h + u] = f2fma(f2fma(pr, pr, f2mul(pi, pi)), sc2, acc[0][4 * h + u]);
                    acc[1][4 * h + u] = f2fma(f2fma(mr, mr, f2mul(mi, mi)), sc2, acc[1][4 * h + u]);
                }
            }
            return true;
        };
        int ecp = beg / T, et = beg - ecp * T, since = 0;   // the image being taken: (channel, pol), time; since a flush
        // after image `item` (local) is taken: add the sums into the accumulator where they must go
        auto taken = [&](int item) {
            ++since;
            const bool wrap = et + 1 == T;
            if (item + 1 == n || wrap || since == a.flush_every) {
                double* dst = a.accum + (size_t)ecp * NP * NP;
                const int iy = ((lane & 16 ? NP - 1 - kk : kk) + NP / 2) & (NP - 1);
#pragma unroll
                for (int m = 0; m < 2; ++m)
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const float2 v = unpack2(acc[m][u]);
                        acc[m][u] = 0ull;
                        const int kx = 16 * qt + 2 * u;
                        const int ix0 = ((m ? NP - 1 - kx : kx) + NP / 2) & (NP - 1);
                        const int ix1 = ((m ? NP - 2 - kx : kx + 1) + NP / 2) & (NP - 1);
                        atomicAdd(dst + iy * NP + ix0, (double)v.x);
                        atomicAdd(dst + iy * NP + ix1, (double)v.y);
                    }
                since = 0;
            }
            et = wrap ? 0 : et + 1;
            ecp += wrap ? 1 : 0;
        };

        bool ok = true;
#pragma unroll 1
        for (int i = -1; i < n; ++i) {
            if (i + 1 < n) {
                if (!(ok = warp_wait(MB_ST1 + ((i + 1) & 1), (i + 1) >> 1))) break;
                fence_after();
                split((i + 1) & 1);
            }
            if (i < 0) continue;
            if (!(ok = epilogue(i >> 1, i & 1))) break;
            taken(i);
        }
        if (!ok) *s_fail = 1;
    } else {
        // the gridding warps and the issuer: one instruction for all of them, since the last warpgroup holds both and a
        // warpgroup's four warps have to execute the same setmaxnreg
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" :: "n"(kRegsOther));
        if (warp < NXW + NGW) {
            // ------------------------------- gridding warps -------------------------------
            const int gw = warp - NXW, gt = tid - 32 * NXW;   // among the gridding warps and threads
            // ---- decode ----
            // voltage row of item (cp, t); for XP, cp = 4 c + v runs over the virtual pols of channel
            // c and the row is pol X of channel c (pol Y for v = 1), the Y row following it
            auto vrow = [&](int cp, int t) -> const VT* {
                if constexpr (XP) {
                    const int c = cp >> 2, p = (cp & 3) == 1 ? 1 : 0;
                    return V + ((long long)t * (a.n_cp >> 1) + 2 * c + p) * (long long)A;
                } else {
                    return V + ((long long)t * a.n_cp + cp) * (long long)A;
                }
            };
            // gains of an antenna for (channel, pol) cp; XP: virtual pol v = cp & 3: X, Y, X + Y, X + iY,
            // gy = phi_v g_Y (phi_2 = 1, phi_3 = i)
            auto gain_of = [&](int cp, int aa, float2& gx, float2& gy) {
                if constexpr (XP) {
                    const int c = cp >> 2, v = cp & 3, p = v == 1 ? 1 : 0;
                    gx = a.gains ? __ldg(a.gains + (size_t)(2 * c + p) * A + aa) : make_float2(1.f, 0.f);
                    gy = a.gains ? __ldg(a.gains + (size_t)(2 * c + 1) * A + aa) : make_float2(1.f, 0.f);
                    if (v == 3) gy = make_float2(-gy.y, gy.x);
                } else {
                    gx = a.gains ? __ldg(a.gains + (size_t)cp * A + aa) : make_float2(1.f, 0.f);
                }
            };
            // Thread gt decodes image gt mod 2 of a pair, antennas gt / 2 + NGT / 2 i.
            const int img_d = gt & 1, ant0 = gt >> 1;
            constexpr int ASTEP = NGT / 2;
            constexpr int VPT = 2;                          // antennas per thread loaded a pair ahead
            int dcp = beg / T, dt = beg - dcp * T;          // (channel*pol, time) of the next pair's first image
            int gcp = -1;                                   // (channel, pol) of the powers summed
            int g0cp = -1;                                  // (channel, pol) of the gains held
            float2 g0[VPT] = {}, gy0[VPT] = {};
            auto next_image = [&](int& cp, int& t) {
                if (++t == T) {
                    t = 0;
                    ++cp;
                }
            };
            // raw voltages of the thread's first antennas for the next pair of images, loaded a pair ahead so that
            // the decode does not wait on HBM; further antennas are loaded when decoded
            VT raw[VPT] = {}, rawy[VPT] = {};
            auto prefetch = [&](int left) {                 // images left from (dcp, dt) on
                int cp = dcp, t = dt;
                if (img_d) next_image(cp, t);
                if (img_d < left) {
                    const VT* base = vrow(cp, t) + ant0;
#pragma unroll
                    for (int i = 0; i < VPT; ++i) {
                        if (ant0 + ASTEP * i < A) {
                            raw[i] = __ldg(base + ASTEP * i);
                            if constexpr (XP) {
                                if ((cp & 3) >= 2) rawy[i] = __ldg(base + A + ASTEP * i);
                            }
                        }
                    }
                }
            };
            auto add_power = [&](int cp, int aa, float v) {
                if (a.power != nullptr && cp >= 0) atomicAdd(a.power + (size_t)cp * A + aa, (double)v);
            };
            // decode + gain of pair p into voltage buffer p mod nvb; the even thread of an antenna sums the
            // power of both images (the same thread throughout, so no barrier separates the updates); the
            // largest component magnitudes go to vmax[p mod 16] (positive float bits order like unsigned
            // integers); then the next pair's voltages are prefetched
            auto decode = [&](int p) {
                float2* vb = reinterpret_cast<float2*>(sVB + (nvb == 2 && (p & 1) ? (size_t)A * VBYTES : 0));
                int cp1 = dcp, t1 = dt;                        // the second image
                next_image(cp1, t1);
                const bool both = 2 * p + 1 < n, there = img_d == 0 || both;
                const int cp = img_d ? cp1 : dcp, t = img_d ? t1 : dt;
                if (there && cp != g0cp) {
#pragma unroll
                    for (int i = 0; i < VPT; ++i)
                        if (ant0 + ASTEP * i < A) gain_of(cp, ant0 + ASTEP * i, g0[i], gy0[i]);
                    g0cp = cp;
                }
                const bool two = XP && (cp & 3) >= 2;          // virtual pol combining X and Y
                float m = 0.f;
                auto one = [&](int aa, VT r, VT ry, float2 gx, float2 gy) {
                    float2 vp = make_float2(0.f, 0.f);
                    if (there) {
                        vp = cmul(gx, Volt<VDT>::dec(r));
                        if constexpr (XP) {
                            if (two) {
                                const float2 w = cmul(gy, Volt<VDT>::dec(ry));
                                vp.x += w.x;
                                vp.y += w.y;
                            }
                        }
                    }
                    if constexpr (LP) {
                        const __half2 hv = __floats2half2_rn(vp.x, vp.y);
                        reinterpret_cast<uint32_t*>(vb)[2 * aa + img_d] = *reinterpret_cast<const uint32_t*>(&hv);
                    } else {
                        vb[2 * aa + img_d] = vp;
                    }
                    m = fmaxf(m, fmaxf(fabsf(vp.x), fabsf(vp.y)));
                    return cnorm(vp);
                };
                auto power = [&](int aa, float n0, float n1) {
                    float pw = PW[aa];
                    if (dcp != gcp) {
                        add_power(gcp, aa, pw);
                        pw = 0.f;
                    }
                    pw += n0;
                    if (both && cp1 != dcp) {
                        add_power(dcp, aa, pw);
                        pw = 0.f;
                    }
                    PW[aa] = pw + n1;
                };
                // the warp's lanes walk the antennas together (the even lane needs its neighbour's power)
                auto both_images = [&](int aa, VT r, VT ry, float2 gx, float2 gy) {
                    const float nn = aa < A ? one(aa, r, ry, gx, gy) : 0.f;
                    const float n1 = __shfl_down_sync(0xffffffffu, nn, 1);
                    if (img_d == 0 && aa < A) power(aa, nn, n1);
                };
#pragma unroll
                for (int i = 0; i < VPT; ++i)
                    if (16 * gw + ASTEP * i < A) both_images(ant0 + ASTEP * i, raw[i], rawy[i], g0[i], gy0[i]);
#pragma unroll 1
                for (int a0 = 16 * gw + ASTEP * VPT; a0 < A; a0 += ASTEP) {
                    const int aa = a0 + (lane >> 1);
                    float2 gx = make_float2(1.f, 0.f), gy = gx;
                    VT r{}, ry{};
                    if (there && aa < A) {
                        const VT* base = vrow(cp, t);
                        gain_of(cp, aa, gx, gy);
                        r = __ldg(base + aa);
                        if constexpr (XP) {
                            if (two) ry = __ldg(base + A + aa);
                        }
                    }
                    both_images(aa, r, ry, gx, gy);
                }
                if (16 * gw < A) {
                    const unsigned bits = __float_as_uint(m);
                    const unsigned m0 = __reduce_max_sync(0xffffffffu, img_d ? 0u : bits);
                    const unsigned m1 = __reduce_max_sync(0xffffffffu, img_d ? bits : 0u);
                    if (lane < 2) atomicMax(vmax + 2 * (p & 15) + lane, lane ? m1 : m0);
                }
                // pair p - 8's words: its F has long been taken (stage 1 of pair p - 3 is done, so every transform
                // warp has split pair p - 4), and none decodes pair p + 8 before this warp has decoded pair p
                if (gt < 2) vmax[2 * ((p + 8) & 15) + gt] = 0u;
                gcp = both ? cp1 : dcp;
                next_image(dcp, dt);
                next_image(dcp, dt);
                prefetch(n - 2 * (p + 1));
            };
            auto flush_power = [&]() {
                if (img_d == 0)
                    for (int aa = ant0; aa < A; aa += ASTEP) add_power(gcp, aa, PW[aa]);
            };

            // ---- gridding ----
            float down0 = 1.f, down1 = 1.f;                 // 2^-s of the pair being gridded
            auto scales = [&](int p) {
                down0 = __uint_as_float((unsigned)(127 - exponent(p, 0)) << 23);
                down1 = __uint_as_float((unsigned)(127 - exponent(p, 1)) << 23);
            };
            // slot position jj of this warp, of pair p, into E buffer p mod 2
            auto grid = [&](int p, int jj) {
                const unsigned char* vb = sVB + (nvb == 2 && (p & 1) ? (size_t)A * VBYTES : 0);
                __half* sEp = sE + (p & 1) * EBUF;
                const int slot = PER_WARP * gw + jj;
                const int2 sl = ldt<SMT>(tSlot + slot);              // first entry, steps (-1: no slot here)
                if (sl.y < 0) return;
                const uint32_t word = __ldg(g.lane + slot * 32 + lane);
                __half* dst = sEp + (word & 0xffffu);
                if (sl.y == 0) {                                     // no antenna reaches these cells
#pragma unroll
                    for (int i = 0; i < (LP ? 4 : 8); ++i)
                        *reinterpret_cast<uint32_t*>(dst + (i & 1) * EIMG + ((i >> 1) & 1) * NG * NG + (i >> 2) * EPART) = 0u;
                    return;
                }
                const ulonglong2 rt = __ldg(reinterpret_cast<const ulonglong2*>(rot + (word >> 16)));
                float r[2][2] = {}, im[2][2] = {};                   // [image][cell]
                // two steps at a time: both steps' table loads, then their voltage loads, so that two
                // dependent load chains overlap
                auto steps = [&](auto cw_tag, auto n_tag, int e) {   // cw_tag: complex weights (tWim) or not
                    constexpr bool CW = decltype(cw_tag)::value;
                    constexpr int U = decltype(n_tag)::value;
                    float2 w[U], wi[U];
                    float4 v[U];
                    int an[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        w[u] = ldt<SMT>(tWre + e + 32 * u);
                        if constexpr (CW) wi[u] = ldt<SMT>(tWim + e + 32 * u);
                        an[u] = ldt<SMT>(tAnt + e + 32 * u);
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        if constexpr (LP) {
                            const uint2 q = reinterpret_cast<const uint2*>(vb)[an[u]];
                            const float2 va = __half22float2(*reinterpret_cast<const __half2*>(&q.x));
                            const float2 vc = __half22float2(*reinterpret_cast<const __half2*>(&q.y));
                            v[u] = make_float4(va.x, va.y, vc.x, vc.y);
                            // weights rounded to FP16, so that every product is exact in FP32
                            w[u] = make_float2(round_h(w[u].x), round_h(w[u].y));
                            if constexpr (CW) wi[u] = make_float2(round_h(wi[u].x), round_h(wi[u].y));
                        } else {
                            v[u] = reinterpret_cast<const float4*>(vb)[an[u]];
                        }
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u)
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            const float wr = c ? w[u].y : w[u].x;
                            r[0][c] = fmaf(wr, v[u].x, r[0][c]);
                            im[0][c] = fmaf(wr, v[u].y, im[0][c]);
                            r[1][c] = fmaf(wr, v[u].z, r[1][c]);
                            im[1][c] = fmaf(wr, v[u].w, im[1][c]);
                            if constexpr (CW) {
                                const float wq = c ? wi[u].y : wi[u].x;
                                r[0][c] = fmaf(-wq, v[u].y, r[0][c]);
                                im[0][c] = fmaf(wq, v[u].x, im[0][c]);
                                r[1][c] = fmaf(-wq, v[u].w, r[1][c]);
                                im[1][c] = fmaf(wq, v[u].z, im[1][c]);
                            }
                        }
                };
                auto walk = [&](auto cw_tag) {
                    int e = sl.x + lane, k = sl.y;
                    for (; k >= 2; k -= 2, e += 64) steps(cw_tag, std::integral_constant<int, 2>{}, e);
                    if (k) steps(cw_tag, std::integral_constant<int, 1>{}, e);
                };
                if (tWim) walk(std::true_type{});
                else walk(std::false_type{});
                // rotate by exp(-i pi (x + y) / NP), scale, split and store y, y + 1 as one word
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const unsigned long long dn = f2dup(i ? down1 : down0);
                    const unsigned long long c = f2mul(rt.x, dn), s = f2mul(rt.y, dn);
                    const unsigned long long re = pack2(make_float2(r[i][0], r[i][1])), ii = pack2(make_float2(im[i][0], im[i][1]));
                    const unsigned long long ro = f2fma(re, c, f2mul(ii, s)), io = f2sub(f2mul(ii, c), f2mul(re, s));
                    __half* d = dst + i * EIMG;
                    if constexpr (LP) {
                        *reinterpret_cast<uint32_t*>(d) = half_pair(ro);
                        *reinterpret_cast<uint32_t*>(d + NG * NG) = half_pair(io);
                    } else {
                        uint32_t rh, rl, ih, il;
                        split2(ro, rh, rl);
                        split2(io, ih, il);
                        *reinterpret_cast<uint32_t*>(d) = rh;
                        *reinterpret_cast<uint32_t*>(d + NG * NG) = ih;
                        *reinterpret_cast<uint32_t*>(d + EPART) = rl;
                        *reinterpret_cast<uint32_t*>(d + EPART + NG * NG) = il;
                    }
                }
            };
            bool ok = true;
            if (np > 0) prefetch(n);
#pragma unroll 1
            for (int p = 0; p < np; ++p) {
                // with one voltage buffer, every warp's gridding of pair p - 1 comes first
                if (nvb == 1 && p > 0 && !(ok = warp_wait(MB_EFULL + ((p - 1) & 1), (p - 1) >> 1))) break;
                decode(p);
                warp_arrive(MB_VFULL);
                if (!(ok = warp_wait(MB_VFULL, p))) break;              // every warp has decoded the pair
                scales(p);
                // the E buffer is free once stage 1 of pair p - 2 has read it
                if (p >= 2 && !(ok = warp_wait(MB_EFREE + (p & 1), (p - 2) >> 1))) break;
#pragma unroll 1
                for (int jj = 0; jj < PER_WARP; ++jj) grid(p, jj);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // E^T visible to the tensor cores
                warp_arrive(MB_EFULL + (p & 1));
            }
            if (ok && np > 0) flush_power();
            if (!ok) *s_fail = 1;
        } else {
            // ------------------------------- issuer -------------------------------
            if (lane == 0 && np > 0) {
            const uint64_t dW = sdesc(smem_u32(sW), 1024), dE = sdesc(smem_u32(sE), 1024);
            constexpr int kWLo = 2 * WTAB / 16, kELo = 2 * EPART / 16, kEBuf = 2 * EBUF / 16, kEImg = 2 * EIMG / 16;
            constexpr int NPROD = LP ? 1 : 3;               // hi hi, hi lo, lo hi (LP: hi hi only)
            auto wait = [&](int i, int parity) { return mbar_wait(mb(i), (uint32_t)parity & 1u, a.wait_tries); };
            auto stage2 = [&](int img) {
                constexpr uint32_t id = idesc(128);
                const uint32_t xa = tX + 128 * img;
#pragma unroll
                for (int q = 0; q < NPROD; ++q)
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const uint32_t xop = xa + 16 * k + (q == 2 ? 64 : 0);
                        const uint64_t b = dW + (uint64_t)((q == 1 ? kWLo : 0) + 16 * k);
                        mma_ts(tF, xop, b, id, (q | k) != 0);
                        mma_ts(tF + 128, xop + 8, b, id, (q | k) != 0);
                    }
                commit(mb(MB_F));
            };
            bool ok = true, issued = false;
            // stage 1 of image i, once its pair is gridded
            auto stage1 = [&](int i) -> bool {
                const int j = i >> 1, img = i & 1;
                if (img == 0 && !wait(MB_EFULL + (j & 1), j >> 1)) return false;
                fence_after();
                constexpr uint32_t id1 = idesc(128);
                const uint64_t e0 = dE + (uint64_t)((j & 1) * kEBuf + img * kEImg);
#pragma unroll
                for (int q = 0; q < NPROD; ++q)
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        mma_ss(tX + 128 * img, dW + (uint64_t)((q == 2 ? kWLo : 0) + 16 * k),
                               e0 + (uint64_t)((q == 1 ? kELo : 0) + 16 * k), id1, (q | k) != 0);
                commit(mb(MB_ST1 + img));
                if (img == 1) commit(mb(MB_EFREE + (j & 1)));
                issued = true;
                return true;
            };
            ok = stage1(0) && (n < 2 || stage1(1));   // an odd last pair has no second image
#pragma unroll 1
            for (int i = 0; ok && i < n; ++i) {
                const int j = i >> 1, img = i & 1;
                if (!(ok = wait(MB_XA + img, j))) break;
                if (i > 0 && !(ok = wait(MB_FREE, i - 1))) break;
                fence_after();
                stage2(img);
                if (i + 2 < n) {
                    if (!(ok = wait(MB_F, i))) break;           // stage 2 has read the columns stage 1 overwrites
                    ok = stage1(i + 2);
                }
            }
            // every MMA issued has completed before the tensor memory is released (full limit)
            if (issued) {
                commit(mb(MB_DRAIN));
                mbar_wait(mb(MB_DRAIN), 0);
            }
            if (!ok) *s_fail = 1;
            }
        }
    }

    fence_before();
    __syncthreads();
    if (tid == 0 && *s_fail && n > 0) {
        // a wait ran out: report it in the plan's status word, mark this CTA's first (channel, pol) block
        if (a.status) atomicOr(a.status, kStatusImageTimeout);
        a.accum[(size_t)(beg / T) * NP * NP] = __longlong_as_double(0x7ff8000000000000LL);
    }
    if (warp == 0) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(512) : "memory");
    }
}

}  // namespace dg

// The antennas the form accepts follow from this size against the device's limit: 2,448 of 232,448 bytes, 1,904 for
// cross-polarisation.  It is the documented limit, not the kernel's need: with one voltage buffer that is dg::smem_fixed
// (192 bytes more than here) and 20 bytes an antenna (12 for LP), so it fits wherever this does from 24 antennas on, and
// under 24 antennas on any device that takes 24.
size_t dftgemm_smem_bytes(int n_ant, bool xpol, bool lp) {
    constexpr size_t kFull = 163904, kLp = 81984;
    static_assert(dg::smem_fixed(false) + 24 * dg::ant_bytes(false, 1) <= kFull + 24 * 28 &&
                      dg::smem_fixed(true) + 24 * dg::ant_bytes(true, 1) <= kLp + 24 * 20, "need within the limit");
    return (lp ? kLp : kFull) + (size_t)n_ant * ((xpol ? 36 : 28) - (lp ? 8 : 0));
}

// Operand tables for N_p = 128: two [128][64] K-major FP16 tables (hi parts, then lo parts) of the rows
// C 0..15, S 0..15, C 16..31, S 16..31, ..., C[k][n] + i S[k][n] = exp(+2 pi i n (k + 1/2) / 128), computed in
// float64; then 128 entries of 4 floats, cos and sin of pi s / 128 and pi (s + 1) / 128: (c, c', s, s').
void dftgemm_tables(std::vector<uint16_t>& out) {
    using namespace dg;
    const double pi = 3.14159265358979323846;
    out.assign((size_t)2 * WTAB + NP * 8, 0);
    for (int r = 0; r < NP; ++r) {
        const int k = 16 * (r / 32) + r % 16;
        for (int n = 0; n < NG; ++n) {
            const double ang = pi * double((n * (2 * k + 1)) % (2 * NP)) / double(NP);
            const double v = (r % 32) < 16 ? std::cos(ang) : std::sin(ang);
            const __half hi = __double2half(v);
            const __half lo = __double2half(v - (double)__half2float(hi));
            out[koff(r, n, NG)] = __half_as_ushort(hi);
            out[(size_t)WTAB + koff(r, n, NG)] = __half_as_ushort(lo);
        }
    }
    for (int s = 0; s < NP; ++s) {
        const double a0 = pi * s / NP, a1 = pi * (s + 1) / NP;
        const float f[4] = {float(std::cos(a0)), float(std::cos(a1)), float(std::sin(a0)), float(std::sin(a1))};
        std::memcpy(&out[(size_t)2 * WTAB + 8 * s], f, sizeof(f));
    }
}

// Slot tables of the tensor-core forms' gridding on an ng x ng grid (64 for N_p = 128, 128 for
// N_p = 256).  The word of pair (x, y), y even, lands in shared-memory bank
// 4 (x mod 8) + (y / 2 mod 4) of every E^T table, so the ng^2 / 2 pairs fall into 32 bank
// classes.  Within each class pairs are ranked by entry count (most first,
// ties by position) and slot r takes the r-th pair of every class: its 32 lanes store to 32
// distinct banks, and classes interleave finely enough over the aperture that the r-th pairs
// of all classes have similar counts.  A slot takes max(count) warp steps; slots go to the
// n_warps gridding warps heaviest first, each to the warp with the fewest steps so far among
// those holding fewer than ceil(slots / n_warps) (ties to the lowest warp), so the slowest
// warp's gridding is about the heaviest slot or the mean, whichever is larger.  Warp w walks
// positions w * ceil(slots / n_warps) ..; positions no slot took hold no entries.
bool dftgemm_gather_tables_ng(int ng, int n_warps, const std::vector<int>& cptr, const std::vector<int2>& cent,
                              const std::vector<float>& cwim, std::vector<int2>& lane, std::vector<int>& base,
                              std::vector<float>& wre, std::vector<float>& wim, std::vector<uint16_t>& ant) {
    using tc::koff;
    const int NW = n_warps;
    const int NPAIR = ng * ng / 2, nslot = NPAIR / 32;
    if ((ng != 64 && ng != 128) || NW < 1 || NW > 32) return false;
    const int per_warp = (nslot + NW - 1) / NW;   // positions per warp; those left over stay empty
    for (const int2& c : cent)
        if (c.y < 0 || c.y > 0xffff) return false;
    struct Pair { int cell, c0, cnt, off; };
    std::vector<Pair> pr(NPAIR);
    for (int yp = 0; yp < ng / 2; ++yp)
        for (int x = 0; x < ng; ++x) {
            const int c = 2 * yp * ng + x;
            const int n0 = cptr[c + 1] - cptr[c], n1 = cptr[c + ng + 1] - cptr[c + ng];
            if (n0 + n1 > 0xffff) return false;
            pr[yp * ng + x] = {c, n0, n0 + n1, koff(x, 2 * yp, ng)};
        }
    auto heavier = [&](int u, int v) { return pr[u].cnt > pr[v].cnt; };
    std::vector<std::vector<int>> cls(32);
    for (int q = 0; q < NPAIR; ++q) cls[4 * ((q % ng) & 7) + ((q / ng) & 3)].push_back(q);
    for (auto& c : cls) std::stable_sort(c.begin(), c.end(), heavier);
    std::vector<std::vector<int>> slots(nslot);
    for (int r = 0; r < nslot; ++r) {
        for (int c = 0; c < 32; ++c) slots[r].push_back(cls[c][r]);
        std::stable_sort(slots[r].begin(), slots[r].end(), heavier);   // lanes in rank order
    }
    std::stable_sort(slots.begin(), slots.end(), [&](const std::vector<int>& u, const std::vector<int>& v) {
        return pr[u[0]].cnt > pr[v[0]].cnt;
    });
    std::vector<int> order;
    for (const auto& sl : slots) order.insert(order.end(), sl.begin(), sl.end());
    lane.assign((size_t)NW * per_warp * 32, int2{0, 0});
    base.assign((size_t)NW * per_warp, -1);   // -1: a position no slot takes (skipped by the kernels)
    wre.clear();
    wim.clear();
    ant.clear();
    std::vector<int> held(NW, 0), steps(NW, 0);
    for (int r = 0; r < nslot; ++r) {
        int w = -1;
        for (int v = 0; v < NW; ++v)
            if (held[v] < per_warp && (w < 0 || steps[v] < steps[w])) w = v;
        const int pos = per_warp * w + held[w]++;
        steps[w] += pr[order[32 * r]].cnt;
        const Pair* P[32];
        for (int i = 0; i < 32; ++i) P[i] = &pr[order[32 * r + i]];
        base[pos] = (int)wre.size();
        for (int i = 0; i < 32; ++i)
            lane[(size_t)pos * 32 + i] = int2{(int)((unsigned)P[i]->c0 | ((unsigned)P[i]->cnt << 16)), P[i]->off};
        // Each lane takes its first cell's entries, then its second's; within a cell the order is
        // free (any fixed order is deterministic), so step by step each lane takes, of its cell's
        // remaining entries, one whose antenna shares a shared-memory bank pair (8-byte voltages:
        // antenna mod 16) with as few antennas already read at this step by its half-warp as
        // possible; lanes with the fewest candidates choose first.
        std::vector<int> rem[32][2];
        for (int i = 0; i < 32; ++i) {
            for (int e = cptr[P[i]->cell]; e < cptr[P[i]->cell + 1]; ++e) rem[i][0].push_back(e);
            for (int e = cptr[P[i]->cell + ng]; e < cptr[P[i]->cell + ng + 1]; ++e) rem[i][1].push_back(e);
        }
        for (int k = 0; k < P[0]->cnt; ++k) {
            int n_act = 0;
            while (n_act < 32 && P[n_act]->cnt > k) ++n_act;
            auto cand = [&](int i) -> std::vector<int>& { return rem[i][k < P[i]->c0 ? 0 : 1]; };
            int ord[32], pick[32], load[2][16] = {};
            std::vector<int> seen[2];            // antennas read at this step, per half-warp
            for (int i = 0; i < n_act; ++i) ord[i] = i;
            std::stable_sort(ord, ord + n_act, [&](int u, int v) { return cand(u).size() < cand(v).size(); });
            for (int t = 0; t < n_act; ++t) {
                const int i = ord[t], h = i / 16;
                std::vector<int>& c = cand(i);
                size_t best = 0;
                int best_cost = 1 << 30;
                for (size_t j = 0; j < c.size(); ++j) {
                    const int an = cent[c[j]].y;
                    const bool dup = std::find(seen[h].begin(), seen[h].end(), an) != seen[h].end();
                    const int cost = dup ? -1 : load[h][an & 15];
                    if (cost < best_cost) {
                        best_cost = cost;
                        best = j;
                    }
                }
                pick[i] = c[best];
                c.erase(c.begin() + (long)best);
                const int an = cent[pick[i]].y;
                if (best_cost >= 0) {
                    ++load[h][an & 15];
                    seen[h].push_back(an);
                }
            }
            for (int i = 0; i < n_act; ++i) {
                const int e = pick[i];
                float wv;
                std::memcpy(&wv, &cent[e].x, sizeof(float));
                wre.push_back(wv);
                wim.push_back(cwim[e]);
                ant.push_back((uint16_t)cent[e].y);
            }
        }
    }
    return true;
}

// The builder above on the 64 x 64 grid with 16 warps (one weight per entry): the checker of its slots calls it.
bool dftgemm_gather_tables(const std::vector<int>& cptr, const std::vector<int2>& cent, const std::vector<float>& cwim,
                           std::vector<int2>& lane, std::vector<int>& base, std::vector<float>& wre,
                           std::vector<float>& wim, std::vector<uint16_t>& ant) {
    return dftgemm_gather_tables_ng(dg::NG, 16, cptr, cent, cwim, lane, base, wre, wim, ant);
}

// Slot tables of the N_p = 128 kernel: as above on the 64 x 64 grid with 11 warps, but an entry is an
// antenna of the cell pair with its weights on both cells (w.x on (x, y), w.y on (x, y + 1), 0 where it
// has none), so a lane's list holds each antenna of its pair once.  A slot's steps hold 32 entries each: a
// lane whose list has ended gets zero weights and an antenna another lane reads at that step.  The order
// of a lane's entries spreads the antennas read at one step over the banks of the 16-byte voltages (8
// lanes at a time, antenna mod 8).
bool dftgemm_pair_tables(const std::vector<int>& cptr, const std::vector<int2>& cent, const std::vector<float>& cwim,
                         std::vector<uint32_t>& lane, std::vector<int2>& slot, std::vector<float2>& w,
                         std::vector<float2>& wim, std::vector<uint16_t>& ant) {
    using tc::koff;
    constexpr int ng = dg::NG, NPAIR = ng * ng / 2, NW = dg::NGW, per_warp = dg::PER_WARP;
    static_assert(dg::NSLOT * 32 == NPAIR, "slots of 32 pairs");
    for (const int2& c : cent)
        if (c.y < 0 || c.y > 0xffff) return false;
    struct Entry { int ant; float2 w, wi; };
    struct Pair { int off, s; std::vector<Entry> e; };
    std::vector<Pair> pr(NPAIR);
    for (int yp = 0; yp < ng / 2; ++yp)
        for (int x = 0; x < ng; ++x) {
            const int c = 2 * yp * ng + x;
            if (cptr[c + 1] - cptr[c] + cptr[c + ng + 1] - cptr[c + ng] > 0xffff) return false;
            Pair& p = pr[yp * ng + x];
            p.off = koff(x, 2 * yp, ng);
            p.s = x + 2 * yp;
            // both cells' entries are in antenna order, each antenna once per cell
            int i = cptr[c], j = cptr[c + ng];
            const int i1 = cptr[c + 1], j1 = cptr[c + ng + 1];
            while (i < i1 || j < j1) {
                const int ai = i < i1 ? cent[i].y : 1 << 30, aj = j < j1 ? cent[j].y : 1 << 30;
                Entry e{ai < aj ? ai : aj, make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                if (ai == e.ant) {
                    std::memcpy(&e.w.x, &cent[i].x, sizeof(float));
                    e.wi.x = cwim[i++];
                }
                if (aj == e.ant) {
                    std::memcpy(&e.w.y, &cent[j].x, sizeof(float));
                    e.wi.y = cwim[j++];
                }
                p.e.push_back(e);
            }
        }
    auto heavier = [&](int u, int v) { return pr[u].e.size() > pr[v].e.size(); };
    std::vector<std::vector<int>> cls(32), slots(dg::NSLOT);
    for (int q = 0; q < NPAIR; ++q) cls[4 * ((q % ng) & 7) + ((q / ng) & 3)].push_back(q);
    for (auto& c : cls) std::stable_sort(c.begin(), c.end(), heavier);
    for (int r = 0; r < dg::NSLOT; ++r) {
        for (int c = 0; c < 32; ++c) slots[r].push_back(cls[c][r]);
        std::stable_sort(slots[r].begin(), slots[r].end(), heavier);   // lanes in rank order
    }
    std::stable_sort(slots.begin(), slots.end(), [&](const std::vector<int>& u, const std::vector<int>& v) {
        return pr[u[0]].e.size() > pr[v[0]].e.size();
    });
    lane.assign((size_t)dg::NPOS * 32, 0u);
    slot.assign(dg::NPOS, int2{0, -1});   // positions no slot takes: -1 steps
    w.clear();
    wim.clear();
    ant.clear();
    // slots to the warps, heaviest first, each to the warp with the least work so far (a slot's overhead is
    // about that of three steps)
    int held[NW] = {}, steps[NW] = {};
    for (const std::vector<int>& sl : slots) {
        int wp = -1;
        for (int v = 0; v < NW; ++v)
            if (held[v] < per_warp && (wp < 0 || steps[v] < steps[wp])) wp = v;
        const int pos = per_warp * wp + held[wp]++;
        steps[wp] += (int)pr[sl[0]].e.size() + (pr[sl[0]].e.empty() ? 1 : 3);
        const int n_step = (int)pr[sl[0]].e.size();
        slot[pos] = int2{(int)ant.size(), n_step};
        std::vector<Entry> rem[32];
        for (int i = 0; i < 32; ++i) {
            rem[i] = pr[sl[i]].e;
            lane[(size_t)pos * 32 + i] = (uint32_t)pr[sl[i]].off | ((uint32_t)pr[sl[i]].s << 16);
        }
        for (int k = 0; k < n_step; ++k) {
            int n_act = 0, ord[32], load[4][8] = {};
            while (n_act < 32 && (int)pr[sl[n_act]].e.size() > k) ++n_act;
            Entry pick[32];
            std::vector<int> seen[4];            // antennas read at this step, per 8 lanes
            for (int i = 0; i < n_act; ++i) ord[i] = i;
            std::stable_sort(ord, ord + n_act, [&](int u, int v) { return rem[u].size() < rem[v].size(); });
            for (int t = 0; t < n_act; ++t) {
                const int i = ord[t], h = i / 8;
                size_t best = 0;
                int best_cost = 1 << 30;
                for (size_t j = 0; j < rem[i].size(); ++j) {
                    const int an = rem[i][j].ant;
                    const bool dup = std::find(seen[h].begin(), seen[h].end(), an) != seen[h].end();
                    const int cost = dup ? -1 : load[h][an & 7];
                    if (cost < best_cost) {
                        best_cost = cost;
                        best = j;
                    }
                }
                pick[i] = rem[i][best];
                rem[i].erase(rem[i].begin() + (long)best);
                if (best_cost >= 0) {
                    ++load[h][pick[i].ant & 7];
                    seen[h].push_back(pick[i].ant);
                }
            }
            for (int i = 0; i < 32; ++i) {
                // past its list a lane follows the first of its 8 lanes that has an entry, or lane 0
                const Entry& e = i < n_act ? pick[i] : pick[8 * (i / 8) < n_act ? 8 * (i / 8) : 0];
                w.push_back(i < n_act ? e.w : make_float2(0.f, 0.f));
                wim.push_back(i < n_act ? e.wi : make_float2(0.f, 0.f));
                ant.push_back((uint16_t)e.ant);
            }
        }
    }
    return true;
}

cudaError_t launch_dftgemm(int vdt, const FwdArgs& a, const void* wtab, const DgPairGather& g, int n_sm, cudaStream_t st,
                           bool xpol, bool lp) {
    const __half* w = static_cast<const __half*>(wtab);
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
    if (lp && xpol) return cudaErrorInvalidValue;
    // two voltage buffers when they fit, and the gather tables beside them when the whole request fits
    auto need = [&](int nvb) { return dg::smem_fixed(lp) + (size_t)a.n_ant * dg::ant_bytes(lp, nvb); };
    const int nvb = need(2) <= (size_t)optin ? 2 : 1;
    const size_t with_tables = ((need(nvb) + 15) & ~(size_t)15) + dg::table_smem_bytes(g.n_ent, g.wim != nullptr);
    const bool smt = with_tables <= (size_t)optin;
    const size_t smem = smt ? with_tables : need(nvb);
    long long grid = n_sm;
    if (grid > a.n_items) grid = a.n_items;
    switch (vdt * 8 + (smt ? 4 : 0) + (xpol ? 2 : 0) + (lp ? 1 : 0)) {
#define EPIC_DG_CASE(V, S, X, L)                                                                             \
    case V * 8 + S * 4 + X * 2 + L:                                                                          \
        e = ensure_smem<dg::moff_dftgemm_kernel<V, S, X, L>>(smem);                                          \
        if (e != cudaSuccess) return e;                                                                      \
        if (grid > 0) dg::moff_dftgemm_kernel<V, S, X, L><<<(unsigned)grid, dg::NTH, smem, st>>>(a, w, g, nvb);\
        return cudaGetLastError();
        EPIC_DG_CASE(0, 0, 0, 0)
        EPIC_DG_CASE(0, 0, 1, 0)
        EPIC_DG_CASE(0, 0, 0, 1)
        EPIC_DG_CASE(0, 1, 0, 0)
        EPIC_DG_CASE(0, 1, 1, 0)
        EPIC_DG_CASE(0, 1, 0, 1)
        EPIC_DG_CASE(1, 0, 0, 0)
        EPIC_DG_CASE(1, 0, 1, 0)
        EPIC_DG_CASE(1, 0, 0, 1)
        EPIC_DG_CASE(1, 1, 0, 0)
        EPIC_DG_CASE(1, 1, 1, 0)
        EPIC_DG_CASE(1, 1, 0, 1)
        EPIC_DG_CASE(2, 0, 0, 0)
        EPIC_DG_CASE(2, 0, 1, 0)
        EPIC_DG_CASE(2, 0, 0, 1)
        EPIC_DG_CASE(2, 1, 0, 0)
        EPIC_DG_CASE(2, 1, 1, 0)
        EPIC_DG_CASE(2, 1, 0, 1)
#undef EPIC_DG_CASE
        default:
            return cudaErrorInvalidValue;
    }
}

}  // namespace epic
