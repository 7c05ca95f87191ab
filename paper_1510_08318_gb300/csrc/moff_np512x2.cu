// Two-pass form of the MOFF imaging step for N_p = 512 (N_g = 256): the zero-padded 2-D spatial
// transform (Sec. 3 "Spatial Fourier Transform") done as a row pass and a column pass with the
// row-transformed grid staged through device memory, instead of one 16-CTA cluster per image.
//
// The cluster form keeps a 512 x 512 image's row-pass output in the distributed shared memory of
// 16 CTAs; only one such cluster fits a GPC, so 112 of 152 SMs work, each with 8 warps.  Here:
//
//   row pass     (twopass_rows2_kernel) two samples of a sub-array at a time, as packed FP32 pairs (a mapping entry
//                read and an instruction serve both): decode + gain, then the 256 non-zero grid rows in rounds of
//                16: the round's cells gridded into shared memory by 8 warps from a table of cell pairs (x, y),
//                (x, y + 1) balanced over them; per row and parity of kx a 256-point transform (16 threads: 16-point,
//                twiddle, exchange, 16-point; the odd kx of the row times exp(+2 pi i x / 512)); the columns kx and
//                kx + 256 of a row go to the scratch image as one 16-byte store (word_of).  Two CTAs of 256 threads
//                an SM, so that one grids while the other transforms; one CTA of 512 (two rounds) where the
//                antennas' voltages leave no room for two (over 665); over 1,587 one sample at a time
//                (twopass_rows_kernel);
//   column pass  (twopass_cols_kernel) per (block of 32 column pairs kx, kx + 256, range of items): 16 threads per
//                column pair do the same two 256-point transforms along y for both columns at once; the next
//                item's rows come by asynchronous copies meanwhile; |.|^2 is added to FP32 sums in tensor memory (64
//                per thread), added to the FP64 accumulator with atomics when the (sub-array, channel, pol) changes,
//                every flush_every samples and at the end.  No CTA barrier.  Where the items are fewer than the
//                groups of 8 blocks that the SMs hold (19 of 152), blocks of 8 column pairs by 128 threads.
//
// Items (sub-array, channel*pol, time) are processed in chunks that fit the scratch buffer (1 MB of FP32 complex
// per 512 x 512 item), owned by the caller of the launcher (a plan or a batch).
//
// Bound by the scratch's way through L2 and DRAM (1.28 GB a chunk of 608 in 421 us: 3.0 TB/s) together with the
// latency of the transforms' exchanges (4 warps a scheduler, 36 % of the issue slots used).  Measured, us, row and
// column pass of a chunk of 608 samples of 400 antennas (22 k mapping entries): 174 and 247; a scalar transform of
// one sample at a time, 32 blocks of 16 columns and plain loads took 160 and 289, and 603 for the row pass of
// 337 k mapping entries.  Whole calls, before and now: 808 samples of 400 antennas 670 and 632; 152 samples of 1,600
// antennas 219 and 187; one sample of 400 73 and 31; 12 sub-arrays on mixed grids, 512 x 512 of up to 337 k entries
// among them, 6,800 and 5,115.
#include <algorithm>
#include <cstring>
#include <type_traits>
#include <vector>
#include "fft_pair.cuh"
#include "tcgen05.cuh"
#include "moff_common.cuh"

namespace epic {
namespace tp {

constexpr int NP = 512, NG = 256;
using G = Geo<512>;                      // S = 16, R1 = 32, NI = 16, KP = 2, twiddle layout
constexpr int S = G::S, R1 = G::R1, NI = G::NI, KP = G::KP;
constexpr int NT = 256;                  // threads per CTA: 16 transforms of 16 threads
constexpr int LANES = NT / S;            // transforms in flight per CTA (rows or columns)
constexpr int RXS = G::RXS;              // exchange row stride (float2)
constexpr size_t ITEM_F2 = (size_t)NG * NP;   // scratch float2 per item (1 MB)
constexpr int VPT = 2;
constexpr int PARTS = 4;                 // of an item's rows, so that few items occupy the chip
static_assert(S == 16 && R1 == 32 && KP == 2, "the 512-point factorisation of the cluster form");

constexpr size_t rows_smem_bytes(int max_ant) {
    return sizeof(float2) * ((size_t)LANES * RXS + G::TWN) + (size_t)max_ant * (2 * sizeof(float2) + sizeof(float));
}

// The two-sample row pass and the column pass: 256-point transforms of 16 threads x 16 values.
constexpr int NT2 = 512, S2 = 16;
constexpr int ROUND = 16;                                   // the gridding's rounds: 16 rows, 8 warps
constexpr size_t kTw = 2 * 256 * sizeof(float2);
constexpr size_t rows2_smem_bytes(int threads, int max_ant) {
    return (size_t)threads / S2 * NG * (sizeof(float4) + sizeof(unsigned long long)) + kTw +
           (size_t)max_ant * (sizeof(float4) + sizeof(float));
}
// the column pass: exchange, the next item's rows (16 words a thread), tables, the tensor-memory address
constexpr size_t cols_smem_bytes(int threads) {
    return (size_t)threads * 16 * (sizeof(unsigned long long) + sizeof(float4)) + kTw + 16;
}
// tables: TW[k2][n1] = exp(+2 pi i n1 k2 / 256), MW[n] = exp(+2 pi i n / 512)
__device__ __forceinline__ void load_tables(float2* TW, float2* MW, const float2* tw, int tid, int threads) {
    for (int i = tid; i < 256; i += threads) {
        TW[i] = tw[(2 * (i >> 4) * (i & 15)) & (NP - 1)];
        MW[i] = tw[i];
    }
}
__device__ __forceinline__ P2 mul_w(const P2& x, float2 w) {
    const unsigned long long c = f2dup(w.x), s = f2dup(w.y), n = f2dup(-w.y);
    return P2{f2fma(x.re, c, f2mul(x.im, n)), f2fma(x.re, s, f2mul(x.im, c))};
}
// z[k1] = sum over the 256 values of the transform's 16 threads, x[n2] = value n1 + 16 n2 (times MW for par = 1), at
// k = n1 + 16 k1 of a 256-point transform: output par + 2 k of the half-zero 512-point one.  rx: the transform's
// 256 words; its threads are the lanes of a half-warp.
// taken() runs once the warp's x are no longer needed.
template <class F>
__device__ __forceinline__ void fft256(P2 (&x)[16], P2 (&z)[16], int n1, int par, const float2* TW, const float2* MW,
                                       unsigned long long* rx, F taken) {
    if (par) {
#pragma unroll
        for (int n2 = 0; n2 < 16; ++n2) {
            x[n2] = mul_w(x[n2], MW[n1 + 16 * n2]);
            if (n2 % 4 == 3) asm volatile("" ::: "memory");   // keeps the compiler from holding every twiddle at once
        }
    }
    dft2<16, +1>(x);
#pragma unroll
    for (int k2 = 1; k2 < 16; ++k2) {
        x[k2] = mul_w(x[k2], TW[16 * k2 + n1]);
        if (k2 % 4 == 3) asm volatile("" ::: "memory");
    }
#pragma unroll
    for (int k2 = 0; k2 < 16; ++k2) rx[16 * k2 + (n1 ^ k2)] = x[k2].re;
    __syncwarp();
    taken();
#pragma unroll
    for (int i = 0; i < 16; ++i) z[i].re = rx[16 * n1 + (i ^ n1)];
    __syncwarp();
#pragma unroll
    for (int k2 = 0; k2 < 16; ++k2) rx[16 * k2 + (n1 ^ k2)] = x[k2].im;
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 16; ++i) z[i].im = rx[16 * n1 + (i ^ n1)];
    __syncwarp();
    dft2<16, +1>(z);
}

// Place of the column pair kx, kx + 256 (kx < 256): the order in which the row pass's threads hold them.  The
// scratch image holds the word of (place, row y) in blocks of KB places by 256 rows, [place / KB][y][place % KB]: a
// warp of the row pass (two rows, 16 adjacent places) stores two runs of 256 bytes; one of the column pass (two
// places, 16 rows) reads whole 32-byte sectors, the rest of whose lines its neighbours read.  Measured, 608 samples
// (us, row pass by CTAs of 512 threads and column pass), KB = 1: 283 and 196, 2: 226 and 239, 4: 201 and 245, 8: 195
// and 248.
__device__ __forceinline__ int place_of(int kx) { return 128 * (kx & 1) + (kx >> 1); }
__device__ __forceinline__ int kx_of(int place) { return (place >> 7) + 2 * (place & 127); }
constexpr int KB = 8;
__device__ __forceinline__ int word_of(int place, int y) { return ((place / KB) * NG + y) * KB + place % KB; }

// sub-array (segment) of global item g, starting the search at s
__device__ __forceinline__ int seg_of(const SegList& L, int g, int s) {
    while (s + 1 < L.n_seg && L.first[s + 1] <= g) ++s;
    return s;
}

// One sample at a time, for the antennas that the two-sample form has no room for (its voltages and powers take 20
// bytes an antenna beside 196 KB).  A quarter of an item's rows is a unit: with whole items 24 samples of 1,600
// antennas took 160 us, column pass included, now 102.
template <int VDT>
__global__ void __launch_bounds__(NT, 2) twopass_rows_kernel(const __grid_constant__ SegList L, int item0, int item1,
                                                             float4* __restrict__ scratch) {
    using VT = typename Volt<VDT>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* RX = reinterpret_cast<float2*>(smem_raw);          // [LANES][RXS]
    float2* TW = RX + LANES * RXS;                             // [S][TWS]
    float2* VB = TW + G::TWN;                                  // [A] g_a V_a
    float2* GN = VB + L.max_ant;                               // [A] gains
    float* PW = reinterpret_cast<float*>(GN + L.max_ant);      // [A] partial sums |g V|^2

    const int tid = threadIdx.x, lane = tid & 31;
    const int n1 = lane % S, r = tid / S;
    G::load_twiddles(TW, L.seg[0].twiddle, tid, NT);
    for (int aa = tid; aa < L.max_ant; aa += NT) PW[aa] = 0.f;

    // units (item, part of its rows), parts fastest: this CTA's contiguous share of the chunk's
    const int units = (item1 - item0) * PARTS;
    const int beg = (int)((long long)units * blockIdx.x / gridDim.x);
    const int end = (int)((long long)units * (blockIdx.x + 1) / gridDim.x);
    if (beg == end) return;
    const int last = item0 + (end - 1) / PARTS;                // its last item
    int sg = seg_of(L, item0 + beg / PARTS, 0), cur_sg = -1, cur_cp = -1, cur = -1;
    VT raw[VPT];
    auto prefetch = [&](int g) {
        const int s = seg_of(L, g, sg);
        const FwdArgs& p = L.seg[s];
        const int li = g - L.first[s], cp = li / p.n_time, t = li - cp * p.n_time;
        const VT* base = static_cast<const VT*>(p.volt) + ((long long)t * p.n_cp + cp) * (long long)p.n_ant;
#pragma unroll
        for (int i = 0; i < VPT; ++i)
            if (tid + NT * i < p.n_ant) raw[i] = __ldg(base + tid + NT * i);
    };
    auto flush_power = [&]() {
        if (cur_sg < 0) return;
        const FwdArgs& p = L.seg[cur_sg];
        for (int aa = tid; aa < p.n_ant; aa += NT) {
            if (p.power != nullptr) atomicAdd(p.power + (size_t)cur_cp * p.n_ant + aa, (double)PW[aa]);
            PW[aa] = 0.f;
        }
    };
    prefetch(item0 + beg / PARTS);
#pragma unroll 1
    for (int u = beg; u < end; ++u) {
        const int g = item0 + u / PARTS, part = u % PARTS;
        sg = seg_of(L, g, sg);
        const FwdArgs& a = L.seg[sg];
        if (g != cur) {
            const int li = g - L.first[sg], cp = li / a.n_time, t = li - cp * a.n_time, A = a.n_ant;
            if (sg != cur_sg || cp != cur_cp) {
                flush_power();
                for (int aa = tid; aa < A; aa += NT)
                    GN[aa] = a.gains ? a.gains[(size_t)cp * A + aa] : make_float2(1.f, 0.f);
                cur_sg = sg;
                cur_cp = cp;
            }
            // decode + gain (owner threads; the CTA of the item's first part sums the powers), prefetch the next item
            const VT* base = static_cast<const VT*>(a.volt) + ((long long)t * a.n_cp + cp) * (long long)A;
#pragma unroll
            for (int i = 0; i < VPT; ++i) {
                const int aa = tid + NT * i;
                if (aa < A) {
                    const float2 vp = cmul(GN[aa], Volt<VDT>::dec(raw[i]));
                    VB[aa] = vp;
                    if (part == 0) PW[aa] += cnorm(vp);
                }
            }
            for (int aa = tid + NT * VPT; aa < A; aa += NT) {
                const float2 vp = cmul(GN[aa], Volt<VDT>::dec(__ldg(base + aa)));
                VB[aa] = vp;
                if (part == 0) PW[aa] += cnorm(vp);
            }
            if (g < last) prefetch(g + 1);
            cur = g;
            __syncthreads();
        }
        float4* img = scratch + (size_t)(g - item0) * (ITEM_F2 / 2);
        float2* rx = RX + r * RXS;
#pragma unroll 1
        for (int y = NG / PARTS * part + r; y < NG / PARTS * (part + 1); y += LANES) {
            float2 x[NI];
            gather_cells<NI, true>(x, a.cell_ptr, y * NG + n1, S, a.cell_ent, a.cell_wim, VB);
            float2 Y[R1];
            dft_halfzero_in<R1, +1>(x, Y);
            G::twiddle_store(rx, Y, TW, n1);
            __syncwarp();
            float2 z[KP][S];
#pragma unroll
            for (int q = 0; q < KP; ++q) {
                const int k2 = n1 * KP + q;
#pragma unroll
                for (int m = 0; m < S; ++m) z[q][m] = rx[k2 * S + (m ^ n1)];
                dft<S, +1>(z[q]);
            }
            // kx = n1 KP + q + R1 k1 at place 128 q + 16 k1 + n1; kx + 256 is k1 + 8
#pragma unroll
            for (int q = 0; q < KP; ++q) {
                float4* dst = img + word_of(128 * q + n1, y);
#pragma unroll
                for (int k1 = 0; k1 < S / 2; ++k1)
                    __stcg(dst + 16 * NG * k1, make_float4(z[q][k1].x, z[q][k1 + 8].x, z[q][k1].y, z[q][k1 + 8].y));
            }
            __syncwarp();
        }
        __syncthreads();
    }
    flush_power();
}

// Gridding of round rb (rows 16 rb .. + 15) of both samples into E by 8 warps.  A lane takes the cell pairs (x, y),
// (x, y + 1) of its warp's slots one after the other: each step is 32 entries, an antenna with its weights on both
// cells and, at a pair's last step, the pair's place in E.  The warp's steps of the round are one run of the table,
// read kGridAhead steps ahead.
template <bool CW>
__device__ __forceinline__ void grid_round(float4* E, const HalfGather& g, int rb, int warp, int lane,
                                           const float4* VB) {
    const int4 run = __ldg(g.run + rb * 8 + warp);
    const float2* wt = g.w + run.x + lane;
    const float2* wim = CW ? g.wim + run.x + lane : nullptr;
    const uint32_t* key = g.key + run.x + lane;
    float2 w[kGridAhead], wi[CW ? kGridAhead : 1];
    uint32_t ky[kGridAhead];
    auto load = [&](int k) {
#pragma unroll
        for (int u = 0; u < kGridAhead; ++u) {
            w[u] = __ldg(wt + 32 * (k + u));
            ky[u] = __ldg(key + 32 * (k + u));
            if constexpr (CW) wi[u] = __ldg(wim + 32 * (k + u));
        }
    };
    if (run.y > 0) load(0);
#pragma unroll 4
    for (int z = 0; z < run.w; ++z) {
        const int o = __ldg(g.empty + run.z + 32 * z + lane);
        E[o] = E[o + NG] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0;      // (re, re', im, im') of (x, y) and (x, y + 1)
#pragma unroll 1
    for (int k = 0; k < run.y; k += kGridAhead) {
        float2 cw[kGridAhead], ci[CW ? kGridAhead : 1];
        uint32_t ck[kGridAhead];
#pragma unroll
        for (int u = 0; u < kGridAhead; ++u) {
            cw[u] = w[u];
            ck[u] = ky[u];
            if constexpr (CW) ci[u] = wi[u];
        }
        if (k + kGridAhead < run.y) load(k + kGridAhead);
#pragma unroll
        for (int u = 0; u < kGridAhead; ++u) {
            const float4 v = VB[ck[u] & 0xffffu];               // (re, im, re', im')
            s0.x = fmaf(cw[u].x, v.x, s0.x);
            s0.y = fmaf(cw[u].x, v.z, s0.y);
            s0.z = fmaf(cw[u].x, v.y, s0.z);
            s0.w = fmaf(cw[u].x, v.w, s0.w);
            s1.x = fmaf(cw[u].y, v.x, s1.x);
            s1.y = fmaf(cw[u].y, v.z, s1.y);
            s1.z = fmaf(cw[u].y, v.y, s1.z);
            s1.w = fmaf(cw[u].y, v.w, s1.w);
            if constexpr (CW) {
                s0.x = fmaf(-ci[u].x, v.y, s0.x);
                s0.y = fmaf(-ci[u].x, v.w, s0.y);
                s0.z = fmaf(ci[u].x, v.x, s0.z);
                s0.w = fmaf(ci[u].x, v.z, s0.w);
                s1.x = fmaf(-ci[u].y, v.y, s1.x);
                s1.y = fmaf(-ci[u].y, v.w, s1.y);
                s1.z = fmaf(ci[u].y, v.x, s1.z);
                s1.w = fmaf(ci[u].y, v.z, s1.w);
            }
            if (ck[u] & kGridLast) {                            // the same for all lanes
                const int o = (ck[u] >> 16) & 0x7fffu;
                E[o] = s0;
                E[o + NG] = s1;
                s0 = s1 = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
    }
}

// NTR threads: 256, two CTAs an SM, or 512
template <int VDT, int NTR>
__global__ void __launch_bounds__(NTR, NT2 / NTR) twopass_rows2_kernel(const __grid_constant__ SegList L, int item0,
                                                                          int item1, float4* __restrict__ scratch) {
    using VT = typename Volt<VDT>::T;
    constexpr int ROWS = NTR / S2, UNITS = NG / ROWS;          // rows at a time, one or two rounds
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4* E = reinterpret_cast<float4*>(smem_raw);           // [ROWS][NG] both samples: (re, re', im, im')
    unsigned long long* RX = reinterpret_cast<unsigned long long*>(E + ROWS * NG);   // [ROWS][256]
    float2* TW = reinterpret_cast<float2*>(RX + ROWS * 256);
    float2* MW = TW + 256;
    float4* VB = reinterpret_cast<float4*>(MW + 256);          // [A] g_a V_a of both samples
    float* PW = reinterpret_cast<float*>(VB + L.max_ant);      // [A] partial sums |g V|^2
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n1 = tid & 15, row = tid >> 4;
    load_tables(TW, MW, L.seg[0].twiddle, tid, NTR);
    for (int aa = tid; aa < L.max_ant; aa += NTR) PW[aa] = 0.f;

    // units (pair of items, round), rounds fastest; this CTA's contiguous share of the chunk's
    const int units = (item1 - item0 + 1) / 2 * UNITS;
    const int beg = (int)((long long)units * blockIdx.x / gridDim.x);
    const int end = (int)((long long)units * (blockIdx.x + 1) / gridDim.x);
    int cur_sg = -1, cur_cp = -1;
    auto flush_power = [&]() {
        if (cur_sg < 0) return;
        const FwdArgs& p = L.seg[cur_sg];
        for (int aa = tid; aa < p.n_ant; aa += NTR) {
            if (p.power != nullptr) atomicAdd(p.power + (size_t)cur_cp * p.n_ant + aa, (double)PW[aa]);
            PW[aa] = 0.f;
        }
    };
    // decode + gain of item g of segment sg, and of g + 1 when two (else zeros); the powers are summed by
    // the CTA of the pair's first round
    auto decode = [&](int g, int sg, bool two, bool count) {
        const FwdArgs& a = L.seg[sg];
        const int A = a.n_ant;
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {
            const bool there = i == 0 || two;
            const int li = g + (there ? i : 0) - L.first[sg], cp = li / a.n_time, t = li - cp * a.n_time;
            if (there && count && (sg != cur_sg || cp != cur_cp)) {
                flush_power();
                cur_sg = sg;
                cur_cp = cp;
            }
            const VT* base = static_cast<const VT*>(a.volt) + ((long long)t * a.n_cp + cp) * (long long)A;
            for (int aa = tid; aa < A; aa += NTR) {
                float2 v = make_float2(0.f, 0.f);
                if (there) {
                    const float2 gn = a.gains ? __ldg(a.gains + (size_t)cp * A + aa) : make_float2(1.f, 0.f);
                    v = cmul(gn, Volt<VDT>::dec(__ldg(base + aa)));
                    if (count) PW[aa] += cnorm(v);
                }
                reinterpret_cast<float2*>(VB + aa)[i] = v;
            }
        }
    };
    int cur_pair = -1;
#pragma unroll 1
    for (int u = beg, sg = 0; u < end; ++u) {
        const int j = u / UNITS, rb = u - j * UNITS, g0 = item0 + 2 * j;
        sg = seg_of(L, g0, sg);
        // the pair's items together, or one after the other where the second is another sub-array's
        const bool second = g0 + 1 < item1, two = second && g0 + 1 < L.first[sg + 1];
        const int parts = second && !two ? 2 : 1;
#pragma unroll 1
        for (int part = 0; part < parts; ++part) {
            const int g = g0 + part, s = part ? seg_of(L, g, sg) : sg;
            if (j != cur_pair || parts == 2) decode(g, s, two, rb == 0);
            __syncthreads();
            const int round = ROWS / ROUND * rb + (warp >> 3);
            float4* Eh = E + (warp >> 3) * ROUND * NG;
            const HalfGather& hg = L.seg[s].half;
            if (hg.wim) grid_round<true>(Eh, hg, round, warp & 7, lane, VB);
            else grid_round<false>(Eh, hg, round, warp & 7, lane, VB);
            __syncthreads();
            const int y = ROWS * rb + row;
            float4* out = scratch + (size_t)(g - item0) * (ITEM_F2 / 2);
#pragma unroll 1
            for (int par = 0; par < 2; ++par) {
                P2 x[16], z[16];
#pragma unroll
                for (int n2 = 0; n2 < 16; ++n2) {
                    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(E + row * NG + n1 + 16 * n2);
                    x[n2] = P2{v.x, v.y};
                }
                fft256(x, z, n1, par, TW, MW, RX + row * 256, [] {});
                // kx = par + 2 (n1 + 16 k1) at place 128 par + 16 k1 + n1; kx + 256 is k1 + 8
                float4* img = out + word_of(128 * par + n1, y);
#pragma unroll
                for (int k1 = 0; k1 < 8; ++k1) {
                    const float2 r0 = unpack2(z[k1].re), r1 = unpack2(z[k1 + 8].re);
                    const float2 i0 = unpack2(z[k1].im), i1 = unpack2(z[k1 + 8].im);
                    __stcg(img + 16 * NG * k1, make_float4(r0.x, r1.x, i0.x, i1.x));
                    if (two) __stcg(img + ITEM_F2 / 2 + 16 * NG * k1, make_float4(r0.y, r1.y, i0.y, i1.y));
                }
            }
            __syncthreads();
        }
        cur_pair = j;
    }
    flush_power();
}

// NTC threads: 512, or 128 where the items are too few to give every SM a CTA of 512
template <int NTC>
__global__ void __launch_bounds__(NTC, NT2 / NTC) twopass_cols_kernel(const __grid_constant__ SegList L, int item0,
                                                                         int item1, const float4* __restrict__ scratch) {
    constexpr int PAIRS = NTC / S2, NB = NP / 2 / PAIRS;        // column pairs of a CTA, blocks of them (8 or 32)
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned long long* RX = reinterpret_cast<unsigned long long*>(smem_raw);   // [PAIRS][256]
    ulonglong2* ST = reinterpret_cast<ulonglong2*>(RX + PAIRS * 256) + threadIdx.x;   // [16][NTC], this thread's words
    float2* TW = reinterpret_cast<float2*>(RX + PAIRS * 256 + 2 * 16 * NTC);
    float2* MW = TW + 256;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(MW + 256);
    const int tid = threadIdx.x, warp = tid >> 5;
    const int n1 = tid & 15;
    load_tables(TW, MW, L.seg[0].twiddle, tid, NTC);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(tc::smem_u32(tslot)), "r"(NTC / 2) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = *tslot;
    // this thread's 64 columns of its warp's tensor-memory lanes
    const uint32_t tacc = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + 64 * (warp >> 2);
    const float zero32[32] = {};
    tc::tst32(tacc, zero32);
    tc::tst32(tacc + 32, zero32);
    tc::tst_wait();

    const int blk = blockIdx.x % NB, grp = blockIdx.x / NB, n_grp = gridDim.x / NB;
    const int place = PAIRS * blk + (tid >> 4), kx = kx_of(place);   // this thread's columns kx, kx + 256
    const int n = item1 - item0;
    const int beg = item0 + (int)((long long)n * grp / n_grp);
    const int end = item0 + (int)((long long)n * (grp + 1) / n_grp);
    int sg = 0, cur_sg = -1, cur_cp = -1, since = 0;
    auto flush = [&]() {
        if (cur_sg < 0) return;
        double* dst = L.seg[cur_sg].accum + (size_t)cur_cp * NP * NP;
#pragma unroll 1
        for (int par = 0; par < 2; ++par) {
            float v[32];
            tc::tld32(tacc + 32 * par, v);
            tc::tld_wait();
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const int ky = par + 2 * (n1 + 16 * (i >> 1));
                atomicAdd(dst + ((ky + NP / 2) & (NP - 1)) * NP + ((kx + 256 * (i & 1) + NP / 2) & (NP - 1)), (double)v[i]);
            }
            tc::tst32(tacc + 32 * par, zero32);
        }
        tc::tst_wait();
    };
    // a thread's words of an item come by asynchronous copies into its own slots
    const uint32_t slot = tc::smem_u32(ST);
    auto fetch = [&](int g) {
        const float4* src = scratch + (size_t)(g - item0) * (ITEM_F2 / 2) + word_of(place, n1);
#pragma unroll
        for (int n2 = 0; n2 < 16; ++n2)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                         :: "r"(slot + n2 * NTC * 16), "l"(src + KB * 16 * n2) : "memory");
    };
    if (beg < end) fetch(beg);
#pragma unroll 1
    for (int g = beg; g < end; ++g) {
        sg = seg_of(L, g, sg);
        const FwdArgs& a = L.seg[sg];
        const int cp = (g - L.first[sg]) / a.n_time;
        if (sg != cur_sg || cp != cur_cp || since == a.flush_every) {
            flush();
            cur_sg = sg;
            cur_cp = cp;
            since = 0;
        }
        ++since;
        asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll 1
        for (int par = 0; par < 2; ++par) {
            P2 x[16], z[16];
#pragma unroll
            for (int n2 = 0; n2 < 16; ++n2) {
                const ulonglong2 v = ST[n2 * NTC];
                x[n2] = P2{v.x, v.y};
            }
            fft256(x, z, n1, par, TW, MW, RX + (tid >> 4) * 256, [&] {
                if (par && g + 1 < end) fetch(g + 1);
            });
            float v[32];
            tc::tld32(tacc + 32 * par, v);
            tc::tld_wait();
#pragma unroll
            for (int k1 = 0; k1 < 16; ++k1) {
                const float2 s = unpack2(f2fma(z[k1].im, z[k1].im,
                                               f2fma(z[k1].re, z[k1].re, pack2(make_float2(v[2 * k1], v[2 * k1 + 1])))));
                v[2 * k1] = s.x;
                v[2 * k1 + 1] = s.y;
            }
            tc::tst32(tacc + 32 * par, v);
        }
        tc::tst_wait();
    }
    flush();
    tc::fence_before();
    __syncthreads();
    if (warp == 0) {
        tc::fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(NTC / 2) : "memory");
    }
}

}  // namespace tp

size_t twopass_scratch_bytes(int chunk_items) { return (size_t)chunk_items * tp::ITEM_F2 * sizeof(float2); }
size_t twopass_rows_smem_bytes(int max_ant) { return tp::rows_smem_bytes(max_ant); }

bool twopass_rows2_fits(int n_ant, size_t smem_optin) { return tp::rows2_smem_bytes(tp::NT2, n_ant) <= smem_optin; }
void twopass_tables(const std::vector<int>& cptr, const std::vector<int2>& cent, const std::vector<float>& cwim,
                    std::vector<int4>& run, std::vector<float2>& w, std::vector<float2>& wim,
                    std::vector<uint32_t>& key, std::vector<uint16_t>& empty) {
    pair_run_tables(tp::NG, tp::ROUND, tp::NG, 8, 8, cptr, cent, cwim, run, w, wim, key, empty);
}

cudaError_t launch_fwd512_twopass(int vdt, const SegList& L, int n_sm, cudaStream_t st, float2* scratch,
                                  int chunk_items) {
    const int total = L.first[L.n_seg];
    if (total == 0) return cudaSuccess;
    if (!scratch || chunk_items < 1) return cudaErrorInvalidValue;
    // the two-sample row pass where every sub-array has its runs (its antennas fit the shared memory): two CTAs of
    // 256 threads an SM where two fit, else one of 512
    bool two = true;
    for (int s = 0; s < L.n_seg; ++s) two = two && L.seg[s].half.run;
    constexpr size_t kSmSmem = 228 * 1024, kCtaSmem = 1024;    // of an SM, and taken by the system for a CTA
    const int threads = !two ? tp::NT : 2 * (tp::rows2_smem_bytes(256, L.max_ant) + kCtaSmem) <= kSmSmem ? 256 : tp::NT2;
    const size_t rsm = two ? tp::rows2_smem_bytes(threads, L.max_ant) : tp::rows_smem_bytes(L.max_ant);
    const size_t csm = tp::cols_smem_bytes(tp::NT2), csm_few = tp::cols_smem_bytes(128);
    using RowsFn = void (*)(const SegList, int, int, float4*);
    RowsFn rows;
    cudaError_t e;
    auto pick = [&](auto v) {
        constexpr int V = decltype(v)::value;
        if (!two) rows = tp::twopass_rows_kernel<V>, e = ensure_smem<tp::twopass_rows_kernel<V>>(rsm);
        else if (threads == 256) rows = tp::twopass_rows2_kernel<V, 256>, e = ensure_smem<tp::twopass_rows2_kernel<V, 256>>(rsm);
        else rows = tp::twopass_rows2_kernel<V, 512>, e = ensure_smem<tp::twopass_rows2_kernel<V, 512>>(rsm);
    };
    switch (vdt) {
        case 0: pick(std::integral_constant<int, 0>()); break;
        case 1: pick(std::integral_constant<int, 1>()); break;
        case 2: pick(std::integral_constant<int, 2>()); break;
        default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    if ((e = ensure_smem<tp::twopass_cols_kernel<tp::NT2>>(csm)) != cudaSuccess) return e;
    if ((e = ensure_smem<tp::twopass_cols_kernel<128>>(csm_few)) != cudaSuccess) return e;
    // the row pass: 512 threads an SM; the column pass: one CTA of 512 an SM, as whole groups of its 8 blocks of
    // column pairs, or blocks of 8 pairs where the items are fewer than the groups
    int sms = n_sm;
    if (L.max_workers > 0 && sms > L.max_workers) sms = L.max_workers;
    const int workers = tp::NT2 / threads * sms;
    const int groups = sms / 8 > 0 ? sms / 8 : 1;
    float4* img = reinterpret_cast<float4*>(scratch);
    for (int i0 = 0; i0 < total; i0 += chunk_items) {
        const int i1 = i0 + chunk_items < total ? i0 + chunk_items : total;
        const int n = i1 - i0, units = two ? (n + 1) / 2 * (tp::NG * tp::S2 / threads) : n * tp::PARTS;
        rows<<<workers < units ? workers : units, threads, rsm, st>>>(L, i0, i1, img);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if (n >= groups) tp::twopass_cols_kernel<tp::NT2><<<8 * groups, tp::NT2, csm, st>>>(L, i0, i1, img);
        else tp::twopass_cols_kernel<128><<<32 * n, 128, csm_few, st>>>(L, i0, i1, img);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace epic
