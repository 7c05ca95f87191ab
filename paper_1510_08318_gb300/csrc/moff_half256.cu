// MOFF imaging and its adjoint at N_p = 256 (N_g = 128) without clusters: one CTA per half image.
//
// The image columns split by the parity of their frequency, kx = h + 2 c, c = 0 .. 127.  Those of one
// parity need only
//     R_h(y, c) = sum_x (E(y, x) exp(+2 pi i h x / 256)) exp(+2 pi i x c / 128),
// a full 128-point transform of the 128 non-zero cells of a row, so the two halves of an image share no
// transform work: what a 4-CTA cluster exchanged through distributed shared memory (every column needs every
// row) stays in one CTA, and only the gridding is done twice.  The rows split the same way along y: the
// even ky are a 128-point transform of a column, the odd ky one of the column times exp(+2 pi i y / 256).
//
// Unit: (channel*pol, h, time).  A persistent CTA of 512 threads per SM walks a contiguous range, keeping the
// sums of its half image (128 columns x 256 rows, FP32) in tensor memory: 64 columns per thread, read, added to
// and written back once per unit (in registers they would leave half the file for the transforms).
// Per unit:
//   decode + gain   owner thread a % 512; the next unit's voltages are prefetched into registers;
//   gridding        cell pairs in slots balanced over the warps (grid_pairs), into the rows' storage;
//   row pass        8 threads per pair of rows, as packed FP32 pairs (one instruction for both): 16-point
//                   transform of the cells n1 + 8 n2, twiddle, exchange in the rows' own storage, two 8-point
//                   transforms;
//   column pass     8 threads per pair of adjacent columns, as packed FP32 pairs,
//                   for each parity of ky: 16-point transform, twiddle, exchange (real, then imaginary parts
//                   through one buffer), two 8-point transforms, |.|^2 added to the sums.
// Three CTA barriers per unit.
//
// The adjoint walks the same units.  It keeps dL/dI of the half image and one parity's result in tensor
// memory, multiplies F by dL/dI, transforms back along y (both parities add up to the 128 rows, in place) and
// along x, and degrids per antenna from shared memory: the two halves' gradients simply add.
//
// Measured (ms): 331 antennas, FP16, 32,768 images 7.05 with the clusters, 6.04 here; gain calibration of 1,024
// antennas, 2,048 images, image and gradient 1.69 -> 1.40.  On the way, forward: 7.40 with twiddle words 128 bytes
// apart (8-way bank conflicts), 6.12 without, 6.03 with the gridding balanced over the warps instead of each
// thread gathering the cells it transforms (calibration 1.64 -> 1.43).  Of a unit's 30,000 cycles the
// gridding takes a third (its table's way from L2), the rows a fifth, the columns two fifths (shared-memory
// wavefronts: 17,000 a unit).
#include <algorithm>
#include <cstring>
#include <vector>
#include "fft_pair.cuh"
#include "moff_common.cuh"
#include "tcgen05.cuh"

namespace epic {
namespace half256 {

constexpr int NP = 256, NG = 128, NT = 512, S = 8, R1 = 16, KP = 2, VPT = 2;
constexpr int NPAIR = 64;              // column pairs of a half image
constexpr int RBS = 68;                // row stride (16-byte column pairs): 4 mod 8, see col_lane
constexpr int RXS = 132;               // exchange stride of a column pair (8-byte pairs): 4 mod 16
constexpr int ROWF2 = 2 * RBS;         // row stride in float2

constexpr size_t kRB = (size_t)NG * RBS * 16, kRX = (size_t)NPAIR * RXS * 8;
constexpr size_t kTables = 2 * 128 * sizeof(float2);
constexpr size_t kFixed = kRB + kRX + kTables + 16;
constexpr size_t fwd_smem(int n_ant) { return kFixed + (size_t)n_ant * (sizeof(float2) + sizeof(float)); }
constexpr size_t bwd_smem(int n_ant) { return kFixed + (size_t)n_ant * 2 * sizeof(float2); }

// swizzle of the exchange: keeps the writes (one k2, all n1) and the reads (one k2 block) apart
__device__ __forceinline__ int swz(int k2) { return (k2 >> 1) & (S - 1); }

struct Smem {
    float4* RB;        // [NG][RBS] row-transformed grid, column pairs (re, re', im, im')
    unsigned long long* RX;   // [NPAIR][RXS]
    float2* TW;        // [16][8] exp(+2 pi i n1 k2 / 128), k2-major: the 8 n1 of a warp read adjacent words
    float2* MW;        // [128] exp(+2 pi i n / 256)
    uint32_t* tslot;
    unsigned char* rest;
};
__device__ __forceinline__ Smem carve(unsigned char* p) {
    Smem m;
    m.RB = reinterpret_cast<float4*>(p);
    m.RX = reinterpret_cast<unsigned long long*>(p + kRB);
    m.TW = reinterpret_cast<float2*>(p + kRB + kRX);
    m.MW = m.TW + 128;
    m.tslot = reinterpret_cast<uint32_t*>(m.MW + 128);
    m.rest = reinterpret_cast<unsigned char*>(m.tslot + 4);
    return m;
}
// tables from the plan's exp(+2 pi i j / 256), tensor memory of 32 W columns
__device__ __forceinline__ uint32_t setup(const Smem& m, const float2* tw, int cols, int tid) {
    for (int i = tid; i < 128; i += NT) {
        m.TW[i] = tw[(2 * (i >> 3) * (i & 7)) & (NP - 1)];
        m.MW[i] = tw[i];
    }
    if (tid < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(tc::smem_u32(m.tslot)), "r"(cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    return *m.tslot;
}

// x * w and x * conj(w) for both values of a pair.  The twiddle is one 8-byte shared-memory read, duplicated in
// registers: as stored (c, c, s, s) and (-s, -s) words it took a third of the kernel's shared-memory bandwidth.
__device__ __forceinline__ P2 mul_w(const P2& x, float2 w) {
    const unsigned long long c = f2dup(w.x), s = f2dup(w.y), n = f2dup(-w.y);
    return P2{f2fma(x.re, c, f2mul(x.im, n)), f2fma(x.re, s, f2mul(x.im, c))};
}
__device__ __forceinline__ P2 mul_wc(const P2& x, float2 w) {
    const unsigned long long c = f2dup(w.x), s = f2dup(w.y), n = f2dup(-w.y);
    return P2{f2fma(x.re, c, f2mul(x.im, s)), f2fma(x.im, c, f2mul(x.re, n))};
}

// Gridding of the 128 x 128 cells into RB, rows y, y + 1 (y even) as packed pairs: (re, re', im, im') of cell x at
// RB[68 y + x].  A lane takes the cell pairs (x, y), (x, y + 1) of its warp's slots one after the other: each step is
// 32 entries, an antenna with its weights on both cells and, at a pair's last step, the pair's place in RB.  The
// table does not fit beside the transform's buffers and comes from L2 in every unit: the warp's steps are one run
// of it, read kGridAhead steps ahead, in 12 bytes an entry (16 bytes an entry, with the cells that no antenna reaches
// among them, took the kernel's L2 reads to 6 TB/s and a third of its time).
template <bool CW>
__device__ __forceinline__ void grid_pairs(const Smem& m, const HalfGather& g, int tid, const float2* VB) {
    const int lane = tid & 31, warp = tid >> 5;
    const int4 run = __ldg(g.run + warp);                  // first entry, steps (a multiple of kGridAhead), first empty
                                                           // place, slots of empty places
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
    for (int z = 0; z < run.w; ++z) m.RB[__ldg(g.empty + run.z + 32 * z + lane)] = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
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
            const float2 v = VB[ck[u] & 0xffffu];
            s.x = fmaf(cw[u].x, v.x, s.x);
            s.y = fmaf(cw[u].y, v.x, s.y);
            s.z = fmaf(cw[u].x, v.y, s.z);
            s.w = fmaf(cw[u].y, v.y, s.w);
            if constexpr (CW) {
                s.x = fmaf(-ci[u].x, v.y, s.x);
                s.y = fmaf(-ci[u].y, v.y, s.y);
                s.z = fmaf(ci[u].x, v.x, s.z);
                s.w = fmaf(ci[u].y, v.x, s.w);
            }
            if (ck[u] & kGridLast) {                           // the same for all lanes
                m.RB[(ck[u] >> 16) & 0x7fffu] = s;
                s = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
    }
}

// Row pass: R_h of all gridded rows, in place, 8 threads per pair of rows (one packed instruction for both);
// the results of a row are stored as pairs of adjacent columns.
__device__ __forceinline__ void row_pass(const Smem& m, int h, int tid) {
    const int n1 = tid & 7, y = 2 * (tid >> 3);
    ulonglong2* rows = reinterpret_cast<ulonglong2*>(m.RB + y * RBS);   // both rows' storage
    P2 x[R1];
#pragma unroll
    for (int n2 = 0; n2 < R1; ++n2) {
        const ulonglong2 v = rows[n1 + S * n2];
        x[n2] = P2{v.x, v.y};
    }
    __syncwarp();
    if (h) {
#pragma unroll
        for (int n2 = 0; n2 < R1; ++n2) {
            x[n2] = mul_w(x[n2], m.MW[n1 + S * n2]);
            if (n2 % 4 == 3) asm volatile("" ::: "memory");   // keeps the compiler from holding every twiddle at once
        }
    }
    dft2<R1, +1>(x);
#pragma unroll
    for (int k2 = 0; k2 < R1; ++k2) {
        const P2 t = k2 == 0 ? x[0] : mul_w(x[k2], m.TW[k2 * S + n1]);
        rows[k2 * S + (n1 ^ swz(k2))] = make_ulonglong2(t.re, t.im);
        if (k2 % 4 == 3) asm volatile("" ::: "memory");
    }
    __syncwarp();
    P2 z[KP][S];
#pragma unroll
    for (int q = 0; q < KP; ++q) {
#pragma unroll
        for (int i = 0; i < S; ++i) {
            const ulonglong2 v = rows[(n1 * KP + q) * S + (i ^ n1)];
            z[q][i] = P2{v.x, v.y};
        }
        dft2<S, +1>(z[q]);
    }
    __syncwarp();
    // c = k2 + 16 k1, k2 = 2 n1 + q: the two q of one k1 are adjacent columns
#pragma unroll
    for (int k1 = 0; k1 < S; ++k1) {
        const float2 r0 = unpack2(z[0][k1].re), r1 = unpack2(z[1][k1].re);
        const float2 i0 = unpack2(z[0][k1].im), i1 = unpack2(z[1][k1].im);
        m.RB[y * RBS + n1 + S * k1] = make_float4(r0.x, r1.x, i0.x, i1.x);
        m.RB[(y + 1) * RBS + n1 + S * k1] = make_float4(r0.y, r1.y, i0.y, i1.y);
    }
}

// A thread's column pair: the four pairs of a warp x 8 n1, n1 slowest, so that the 8 lanes of a 16-byte
// access are 2 rows x 4 pairs (8 different banks) and those of an 8-byte exchange access 4 n1 x 4 pairs.
__device__ __forceinline__ void col_lane(int tid, int& pair, int& n1) {
    pair = 4 * (tid >> 5) + (tid & 3);
    n1 = (tid >> 2) & 7;
}

// Columns forward, one parity of ky: z[q][k1] = F at ky = par + 2 (2 n1 + q + 16 k1).
__device__ __forceinline__ void col_forward(const Smem& m, int pair, int n1, int par, P2 (&z)[KP][S]) {
    P2 x[R1];
#pragma unroll
    for (int n2 = 0; n2 < R1; ++n2) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(m.RB + (n1 + S * n2) * RBS + pair);
        x[n2] = P2{v.x, v.y};
    }
    if (par) {
#pragma unroll
        for (int n2 = 0; n2 < R1; ++n2) {
            x[n2] = mul_w(x[n2], m.MW[n1 + S * n2]);
            if (n2 % 4 == 3) asm volatile("" ::: "memory");   // keeps the compiler from holding every twiddle at once
        }
    }
    dft2<R1, +1>(x);
    unsigned long long* rx = m.RX + pair * RXS;
#pragma unroll
    for (int k2 = 1; k2 < R1; ++k2) {
        x[k2] = mul_w(x[k2], m.TW[k2 * S + n1]);
        if (k2 % 4 == 3) asm volatile("" ::: "memory");
    }
#pragma unroll
    for (int k2 = 0; k2 < R1; ++k2) rx[k2 * S + (n1 ^ swz(k2))] = x[k2].re;
    __syncwarp();
#pragma unroll
    for (int q = 0; q < KP; ++q)
#pragma unroll
        for (int i = 0; i < S; ++i) z[q][i].re = rx[(n1 * KP + q) * S + (i ^ n1)];
    __syncwarp();
#pragma unroll
    for (int k2 = 0; k2 < R1; ++k2) rx[k2 * S + (n1 ^ swz(k2))] = x[k2].im;
    __syncwarp();
#pragma unroll
    for (int q = 0; q < KP; ++q) {
#pragma unroll
        for (int i = 0; i < S; ++i) z[q][i].im = rx[(n1 * KP + q) * S + (i ^ n1)];
        dft2<S, +1>(z[q]);
    }
    __syncwarp();
}

// Transposed columns of one parity: x[n2] = sum over this parity's ky of z exp(-2 pi i y ky / 256).
__device__ __forceinline__ void col_adjoint(const Smem& m, int pair, int n1, int par, P2 (&z)[KP][S], P2 (&x)[R1]) {
    unsigned long long* rx = m.RX + pair * RXS;
#pragma unroll
    for (int q = 0; q < KP; ++q) {
        dft2<S, -1>(z[q]);
#pragma unroll
        for (int i = 0; i < S; ++i) rx[(n1 * KP + q) * S + (i ^ n1)] = z[q][i].re;
    }
    __syncwarp();
#pragma unroll
    for (int k2 = 0; k2 < R1; ++k2) x[k2].re = rx[k2 * S + (n1 ^ swz(k2))];
    __syncwarp();
#pragma unroll
    for (int q = 0; q < KP; ++q)
#pragma unroll
        for (int i = 0; i < S; ++i) rx[(n1 * KP + q) * S + (i ^ n1)] = z[q][i].im;
    __syncwarp();
#pragma unroll
    for (int k2 = 0; k2 < R1; ++k2) x[k2].im = rx[k2 * S + (n1 ^ swz(k2))];
    __syncwarp();
#pragma unroll
    for (int k2 = 1; k2 < R1; ++k2) {
        x[k2] = mul_wc(x[k2], m.TW[k2 * S + n1]);
        if (k2 % 4 == 3) asm volatile("" ::: "memory");
    }
    dft2<R1, -1>(x);
    if (par) {
#pragma unroll
        for (int n2 = 0; n2 < R1; ++n2) {
            x[n2] = mul_wc(x[n2], m.MW[n1 + S * n2]);
            if (n2 % 4 == 3) asm volatile("" ::: "memory");
        }
    }
}

// Image pixel of value (par, q, k1, comp) of a thread's pair.
__device__ __forceinline__ int pixel(int h, int pair, int n1, int par, int q, int k1, int comp) {
    const int ky = par + 2 * (KP * n1 + q + R1 * k1), kx = h + 2 * (2 * pair + comp);
    return ((ky + NP / 2) & (NP - 1)) * NP + ((kx + NP / 2) & (NP - 1));
}

// unit at cost position c of a list (item_at_cost of the forward kernels, in half images)
__device__ __forceinline__ int unit_at_cost(const SegList& L, long long c) {
    int s = 0;
    while (s + 1 < L.n_seg && L.cost[s + 1] <= c) ++s;
    const long long i = (2 * (c - L.cost[s]) + L.weight[s] - 1) / L.weight[s];
    const long long n = 2LL * (L.first[s + 1] - L.first[s]);
    return (int)(2LL * L.first[s] + (i < n ? i : n));
}

template <int VDT>
__global__ void __launch_bounds__(NT, 1) half256_fwd_kernel(const __grid_constant__ SegList L) {
    using VT = typename Volt<VDT>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Smem m = carve(smem_raw);
    float2* VB = reinterpret_cast<float2*>(m.rest);          // [A] g_a V_a
    float* PW = reinterpret_cast<float*>(VB + L.max_ant);    // [A] partial sums |g V|^2
    const int tid = threadIdx.x, warp = tid >> 5;
    for (int aa = tid; aa < L.max_ant; aa += NT) PW[aa] = 0.f;
    // this thread's 64 columns of its warp's tensor-memory lanes
    const uint32_t tmem = setup(m, L.seg[0].twiddle, 256, tid);
    const uint32_t tacc = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + 64 * (warp >> 2);
    const float zero32[32] = {};
    tc::tst32(tacc, zero32);
    tc::tst32(tacc + 32, zero32);
    tc::tst_wait();
    int pair, n1;
    col_lane(tid, pair, n1);

    const long long total = 2LL * L.first[L.n_seg];
    const int nw = gridDim.x, wid = blockIdx.x;
    auto cut = [&](int w) -> int {
        return L.n_seg == 1 ? (int)(total * w / nw)
                            : unit_at_cost(L, L.cost[L.n_seg] / nw * w + L.cost[L.n_seg] % nw * w / nw);
    };
    const int beg = cut(wid), end = cut(wid + 1);
    int sg = 0;
    while (sg + 1 < L.n_seg && 2 * L.first[sg + 1] <= beg) ++sg;

    // unit u -> (segment, channel*pol, half, time), the half slower than the time
    struct Where { int sg, cp, h, t; };
    auto where = [&](int u, int s) -> Where {
        while (s + 1 < L.n_seg && 2 * L.first[s + 1] <= u) ++s;
        const int li = u - 2 * L.first[s], T = L.seg[s].n_time, ch = li / T;
        return Where{s, ch >> 1, ch & 1, li - ch * T};
    };
    VT raw[VPT];
    float2 gn[VPT];
    auto prefetch = [&](const Where& w) {
        const FwdArgs& a = L.seg[w.sg];
        const VT* base = static_cast<const VT*>(a.volt) + ((long long)w.t * a.n_cp + w.cp) * (long long)a.n_ant;
#pragma unroll
        for (int i = 0; i < VPT; ++i)
            if (tid + NT * i < a.n_ant) raw[i] = __ldg(base + tid + NT * i);
    };
    Where cur{-1, -1, -1, 0};         // of the sums held
    int since = 0;
    auto flush = [&]() {
        const FwdArgs& a = L.seg[cur.sg];
        double* dst = a.accum + (size_t)cur.cp * NP * NP;
#pragma unroll 1
        for (int par = 0; par < 2; ++par) {
            float v[32];
            tc::tld32(tacc + 32 * par, v);
            tc::tld_wait();
#pragma unroll
            for (int i = 0; i < 32; ++i)
                atomicAdd(dst + pixel(cur.h, pair, n1, par, i >> 4, (i >> 1) & 7, i & 1), (double)v[i]);
            tc::tst32(tacc + 32 * par, zero32);
        }
        tc::tst_wait();
        for (int aa = tid; aa < a.n_ant; aa += NT) {
            // both halves see every sample: the first one counts the powers
            if (a.power != nullptr && cur.h == 0) atomicAdd(a.power + (size_t)cur.cp * a.n_ant + aa, (double)PW[aa]);
            PW[aa] = 0.f;
        }
        since = 0;
    };
    // decode + gain of unit w into VB (its voltages are in raw), then prefetch the unit after it
    auto decode = [&](const Where& w, int u) {
        const FwdArgs& a = L.seg[w.sg];
        const int A = a.n_ant;
        const VT* base = static_cast<const VT*>(a.volt) + ((long long)w.t * a.n_cp + w.cp) * (long long)A;
        auto gain = [&](int aa) { return a.gains ? __ldg(a.gains + (size_t)w.cp * A + aa) : make_float2(1.f, 0.f); };
        if (w.sg != cur.sg || w.cp != cur.cp || w.h != cur.h || since == a.flush_every) {
            if (cur.sg >= 0) flush();
#pragma unroll
            for (int i = 0; i < VPT; ++i)
                if (tid + NT * i < A) gn[i] = gain(tid + NT * i);
            cur = w;
        }
        ++since;
#pragma unroll
        for (int i = 0; i < VPT; ++i) {
            const int aa = tid + NT * i;
            if (aa < A) {
                const float2 v = cmul(gn[i], Volt<VDT>::dec(raw[i]));
                VB[aa] = v;
                PW[aa] += cnorm(v);
            }
        }
        for (int aa = tid + NT * VPT; aa < A; aa += NT) {
            const float2 v = cmul(gain(aa), Volt<VDT>::dec(__ldg(base + aa)));
            VB[aa] = v;
            PW[aa] += cnorm(v);
        }
        if (u + 1 < end) prefetch(where(u + 1, w.sg));
    };
    if (beg < end) prefetch(where(beg, sg));
#pragma unroll 1
    for (int u = beg; u < end; ++u) {
        const Where w = where(u, sg);
        sg = w.sg;
        decode(w, u);
        __syncthreads();
        if (L.seg[w.sg].half.wim) grid_pairs<true>(m, L.seg[w.sg].half, tid, VB);
        else grid_pairs<false>(m, L.seg[w.sg].half, tid, VB);
        __syncthreads();
        row_pass(m, w.h, tid);
        __syncthreads();
#pragma unroll 1
        for (int par = 0; par < 2; ++par) {
            P2 z[KP][S];
            col_forward(m, pair, n1, par, z);
            float v[32];
            tc::tld32(tacc + 32 * par, v);
            tc::tld_wait();
#pragma unroll
            for (int q = 0; q < KP; ++q)
#pragma unroll
                for (int k1 = 0; k1 < S; ++k1) {
                    const int i = 16 * q + 2 * k1;
                    const float2 s = unpack2(f2fma(z[q][k1].im, z[q][k1].im,
                                                   f2fma(z[q][k1].re, z[q][k1].re, pack2(make_float2(v[i], v[i + 1])))));
                    v[i] = s.x;
                    v[i + 1] = s.y;
                }
            tc::tst32(tacc + 32 * par, v);
        }
        tc::tst_wait();
        // RB is written again only after the next unit's first barrier, which every warp's column pass precedes
    }
    if (cur.sg >= 0) flush();
    tc::fence_before();
    __syncthreads();
    if (warp == 0) {
        tc::fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(256) : "memory");
    }
}

template <int VDT>
__global__ void __launch_bounds__(NT, 1) half256_bwd_kernel(const BwdArgs a) {
    using VT = typename Volt<VDT>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Smem m = carve(smem_raw);
    const int A = a.n_ant, T = a.n_time;
    float2* VB = reinterpret_cast<float2*>(m.rest);          // [A] g_a V_a
    float2* GA = VB + A;                                     // [A] partial gradient sums
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int aa = tid; aa < A; aa += NT) GA[aa] = make_float2(0.f, 0.f);
    const uint32_t tmem = setup(m, a.twiddle, 512, tid);
    const uint32_t tlane = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + 64 * (warp >> 2);
    const uint32_t tg = tlane, tq = tlane + 256;             // dL/dI of both parities; the even parity's result
    int pair, n1;
    col_lane(tid, pair, n1);

    const long long total = 2 * a.n_items;
    const long long beg = total * blockIdx.x / gridDim.x, end = total * (blockIdx.x + 1) / gridDim.x;
    const VT* V = static_cast<const VT*>(a.volt);
    VT raw[VPT], now[VPT];
    auto vrow = [&](long long u) -> const VT* {
        const int ch = (int)(u / T), t = (int)(u - (long long)ch * T);
        return V + ((long long)t * a.n_cp + (ch >> 1)) * (long long)A;
    };
    auto prefetch = [&](long long u) {
        const VT* base = vrow(u);
#pragma unroll
        for (int i = 0; i < VPT; ++i)
            if (tid + NT * i < A) raw[i] = __ldg(base + tid + NT * i);
    };
    auto flush = [&](int ch) {
        for (int aa = tid; aa < A; aa += NT) {
            float2* dst = a.grad_gains + (size_t)(ch >> 1) * A + aa;
            atomicAdd(&dst->x, a.scale * GA[aa].x);
            atomicAdd(&dst->y, a.scale * GA[aa].y);
            GA[aa] = make_float2(0.f, 0.f);
        }
    };
    if (beg < end) prefetch(beg);
    int cur = -1;                                            // (channel*pol, half) of the sums held
    float2 gn[VPT];
#pragma unroll 1
    for (long long u = beg; u < end; ++u) {
        const int ch = (int)(u / T), cp = ch >> 1, h = ch & 1;
        auto gain = [&](int aa) { return a.gains ? __ldg(a.gains + (size_t)cp * A + aa) : make_float2(1.f, 0.f); };
        if (ch != cur) {
            if (cur >= 0) flush(cur);
            const float* gi = a.grad_image + (size_t)cp * NP * NP;
#pragma unroll 1
            for (int par = 0; par < 2; ++par) {
                float v[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] = __ldg(gi + pixel(h, pair, n1, par, i >> 4, (i >> 1) & 7, i & 1));
                tc::tst32(tg + 32 * par, v);
            }
            tc::tst_wait();
#pragma unroll
            for (int i = 0; i < VPT; ++i)
                if (tid + NT * i < A) gn[i] = gain(tid + NT * i);
            cur = ch;
        }
        // decode; this unit's first voltages stay in registers for the degridding
        const VT* base = vrow(u);
#pragma unroll
        for (int i = 0; i < VPT; ++i) {
            now[i] = raw[i];
            if (tid + NT * i < A) VB[tid + NT * i] = cmul(gn[i], Volt<VDT>::dec(now[i]));
        }
        for (int aa = tid + NT * VPT; aa < A; aa += NT) VB[aa] = cmul(gain(aa), Volt<VDT>::dec(__ldg(base + aa)));
        if (u + 1 < end) prefetch(u + 1);
        __syncthreads();
        if (a.half.wim) grid_pairs<true>(m, a.half, tid, VB);
        else grid_pairs<false>(m, a.half, tid, VB);
        __syncthreads();
        row_pass(m, h, tid);
        __syncthreads();
        // columns: F, times dL/dI, back to the rows; a thread reads and overwrites its own RB elements only
#pragma unroll 1
        for (int par = 0; par < 2; ++par) {
            P2 z[KP][S], x[R1];
            col_forward(m, pair, n1, par, z);
            float v[32];
            tc::tld32(tg + 32 * par, v);
            tc::tld_wait();
#pragma unroll
            for (int q = 0; q < KP; ++q)
#pragma unroll
                for (int k1 = 0; k1 < S; ++k1) {
                    const unsigned long long g = pack2(make_float2(v[16 * q + 2 * k1], v[16 * q + 2 * k1 + 1]));
                    z[q][k1].re = f2mul(z[q][k1].re, g);
                    z[q][k1].im = f2mul(z[q][k1].im, g);
                }
            col_adjoint(m, pair, n1, par, z, x);
#pragma unroll
            for (int half = 0; half < 2; ++half) {           // 8 rows: 32 words
                float w[32];
                if (par) {
                    tc::tld32(tq + 32 * half, w);
                    tc::tld_wait();
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    P2& e = x[8 * half + i];
                    if (par) {
                        e.re = f2add(e.re, pack2(make_float2(w[4 * i], w[4 * i + 1])));
                        e.im = f2add(e.im, pack2(make_float2(w[4 * i + 2], w[4 * i + 3])));
                        *reinterpret_cast<ulonglong2*>(m.RB + (n1 + S * (8 * half + i)) * RBS + pair) = make_ulonglong2(e.re, e.im);
                    } else {
                        const float2 r = unpack2(e.re), j = unpack2(e.im);
                        w[4 * i] = r.x;
                        w[4 * i + 1] = r.y;
                        w[4 * i + 2] = j.x;
                        w[4 * i + 3] = j.y;
                    }
                }
                if (!par) tc::tst32(tq + 32 * half, w);
            }
            if (!par) tc::tst_wait();
        }
        __syncthreads();
        // transposed rows: Q_h(y, x) of the 128 cells of each row, into the row's storage as float2
#pragma unroll 1
        for (int rnd = 0; rnd < 2; ++rnd) {
            const int y = 64 * rnd + (tid >> 3), r1 = lane & 7;
            float2* row = reinterpret_cast<float2*>(m.RB + y * RBS);
            float2 z[KP][S];
#pragma unroll
            for (int k1 = 0; k1 < S; ++k1) {
                const float4 f = m.RB[y * RBS + r1 + S * k1];
                z[0][k1] = make_float2(f.x, f.z);
                z[1][k1] = make_float2(f.y, f.w);
            }
            __syncwarp();
#pragma unroll
            for (int q = 0; q < KP; ++q) {
                dft<S, -1>(z[q]);
#pragma unroll
                for (int i = 0; i < S; ++i) row[(r1 * KP + q) * S + (i ^ r1)] = z[q][i];
            }
            __syncwarp();
            float2 x[R1];
            x[0] = row[r1 ^ swz(0)];
#pragma unroll
            for (int k2 = 1; k2 < R1; ++k2) {
                x[k2] = cmulc(row[k2 * S + (r1 ^ swz(k2))], m.TW[k2 * S + r1]);
            }
            dft<R1, -1>(x);
            __syncwarp();
#pragma unroll
            for (int n2 = 0; n2 < R1; ++n2) {
                row[r1 + S * n2] = h ? cmulc(x[n2], m.MW[r1 + S * n2]) : x[n2];
            }
        }
        __syncthreads();
        // degrid: per antenna, sum_g conj(M[g, a]) Q_h(g), times conj(V_a)
        const float2* Q = reinterpret_cast<const float2*>(m.RB);
        auto degrid = [&](int aa, float2 v) {
            float2 s = make_float2(0.f, 0.f);
            const int e1 = __ldg(a.half.ant_ptr + aa + 1);
#pragma unroll 4
            for (int e = __ldg(a.half.ant_ptr + aa); e < e1; ++e) {
                const int2 en = __ldg(a.half.ant_ent + e);
                const float2 qv = Q[en.y];
                // conj(w) * q
                const float wr = __int_as_float(en.x), wi = a.half.ant_wim ? __ldg(a.half.ant_wim + e) : 0.f;
                s.x = fmaf(wr, qv.x, fmaf(wi, qv.y, s.x));
                s.y = fmaf(wr, qv.y, fmaf(-wi, qv.x, s.y));
            }
            // conj(v) * s
            GA[aa].x += v.x * s.x + v.y * s.y;
            GA[aa].y += v.x * s.y - v.y * s.x;
        };
#pragma unroll
        for (int i = 0; i < VPT; ++i)
            if (tid + NT * i < A) degrid(tid + NT * i, Volt<VDT>::dec(now[i]));
        for (int aa = tid + NT * VPT; aa < A; aa += NT) degrid(aa, Volt<VDT>::dec(__ldg(base + aa)));
        // the next unit's rows are written after its first barrier
    }
    if (cur >= 0) flush(cur);
    tc::fence_before();
    __syncthreads();
    if (warp == 0) {
        tc::fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(512) : "memory");
    }
}

template <int VDT>
cudaError_t launch_fwd(const SegList& L, int n_sm, cudaStream_t st) {
    const size_t smem = fwd_smem(L.max_ant);
    const cudaError_t e = ensure_smem<half256_fwd_kernel<VDT>>(smem);
    if (e != cudaSuccess) return e;
    long long grid = n_sm;
    if (L.max_workers > 0 && grid > L.max_workers) grid = L.max_workers;
    if (grid > 2LL * L.first[L.n_seg]) grid = 2LL * L.first[L.n_seg];
    if (grid == 0) return cudaSuccess;
    half256_fwd_kernel<VDT><<<(unsigned)grid, NT, smem, st>>>(L);
    return cudaGetLastError();
}

template <int VDT>
cudaError_t launch_bwd(const BwdArgs& a, int n_sm, cudaStream_t st) {
    const size_t smem = bwd_smem(a.n_ant);
    const cudaError_t e = ensure_smem<half256_bwd_kernel<VDT>>(smem);
    if (e != cudaSuccess) return e;
    const long long grid = 2 * a.n_items < n_sm ? 2 * a.n_items : n_sm;
    if (grid == 0) return cudaSuccess;
    half256_bwd_kernel<VDT><<<(unsigned)grid, NT, smem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace half256

// Gridding runs of the kernels that walk cell pairs (here and in the two-pass 512 x 512 form): an ng x ng grid in
// rounds of `rows` rows (a round's place of cell (x, y) is stride (y mod rows) + x), each shared out to `warps`
// warps (at most 16); an antenna's voltage is a shared-memory word of 128 / per bytes.  The 16-byte word of (x, y),
// y even, lies in bank group x mod 8, so a round's pairs fall into 8 classes; in each they are ranked by entry count
// (most first) and slot r takes ranks 4 r to 4 r + 3 of every class, so that the lanes of a quarter-warp store to 8
// different bank groups and a slot's pairs have similar counts.
void pair_run_tables(int ng, int rows, int stride, int warps, int per, const std::vector<int>& cptr, const std::vector<int2>& cent,
                     const std::vector<float>& cwim, std::vector<int4>& run, std::vector<float2>& w, std::vector<float2>& wim,
                     std::vector<uint32_t>& key, std::vector<uint16_t>& empty) {
    constexpr int MAXW = 16;
    const int NG = ng, NSLOT = rows * ng / 64, NPAIR = rows * ng / 2;
    struct Entry { int ant; float2 w, wi; };
    const float2 none = make_float2(0.f, 0.f);
    // by decreasing value, equal values in their order
    std::vector<int> first, sorted;
    auto by_decreasing = [&](std::vector<int>& v, const std::vector<int>& value) {
        int most = 0;
        for (int q : v) most = std::max(most, value[q]);
        first.assign((size_t)most + 2, 0);
        for (int q : v) ++first[most - value[q] + 1];
        for (int i = 0; i <= most; ++i) first[i + 1] += first[i];
        sorted.resize(v.size());
        for (int q : v) sorted[first[most - value[q]]++] = q;
        v.swap(sorted);
    };
    run.clear();
    w.reserve(w.size() + cent.size());
    wim.reserve(wim.size() + cent.size());
    key.reserve(key.size() + cent.size());
    std::vector<Entry> all;                                  // the round's entries, pair by pair
    std::vector<int> beg(NPAIR), cnt(NPAIR), cls[8], steps(NSLOT), order(NSLOT), mine[MAXW];
    for (int rb = 0; rb < ng / rows; ++rb) {
        all.clear();
        for (auto& c : cls) c.clear();
        for (int q = 0; q < NPAIR; ++q) {
            const int c = (rb * rows + 2 * (q / NG)) * NG + q % NG;
            beg[q] = (int)all.size();
            int i = cptr[c], j = cptr[c + NG];               // both in antenna order
            while (i < cptr[c + 1] || j < cptr[c + NG + 1]) {
                const int ai = i < cptr[c + 1] ? cent[i].y : 1 << 30, aj = j < cptr[c + NG + 1] ? cent[j].y : 1 << 30;
                Entry e{std::min(ai, aj), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                if (ai == e.ant) {
                    std::memcpy(&e.w.x, &cent[i].x, sizeof(float));
                    e.wi.x = cwim[i++];
                }
                if (aj == e.ant) {
                    std::memcpy(&e.w.y, &cent[j].x, sizeof(float));
                    e.wi.y = cwim[j++];
                }
                all.push_back(e);
            }
            cnt[q] = (int)all.size() - beg[q];
            cls[q & 7].push_back(q);                         // ng is a multiple of 8
        }
        for (auto& c : cls) by_decreasing(c, cnt);
        for (int r = 0; r < NSLOT; ++r) {
            order[r] = r;
            steps[r] = 0;
            for (auto& c : cls) steps[r] = std::max(steps[r], cnt[c[4 * r]]);
        }
        by_decreasing(order, steps);
        // slots to the warps, heaviest first, each to the warp with the fewest steps (one for a slot that no antenna
        // reaches: its zeros are stored all the same)
        int load[MAXW] = {};
        for (auto& v : mine) v.clear();
        for (int r : order) {
            const int wp = (int)(std::min_element(load, load + warps) - load);
            mine[wp].push_back(r);
            load[wp] += std::max(1, steps[r]);
        }
        for (int wp = 0; wp < warps; ++wp) {
            run.push_back(int4{(int)key.size(), 0, (int)empty.size(), 0});
            int4& me = run.back();
            for (int r : mine[wp]) me.y += steps[r];
            me.y = (me.y + kGridAhead - 1) / kGridAhead * kGridAhead;
            size_t out = key.size();
            // the steps past the last pair's keep zero weights, and an antenna (a run that is not empty has entries)
            w.resize(out + 32 * (size_t)me.y, none);
            wim.resize(w.size(), none);
            key.resize(w.size(), me.y ? (uint32_t)cent[0].y : 0u);
            for (int r : mine[wp]) {
                Entry* rem[32];                              // a lane's remaining entries, in antenna order
                int left[32];
                uint32_t off[32];
                for (int l = 0; l < 32; ++l) {
                    const int q = cls[l & 7][4 * r + l / 8];
                    rem[l] = all.data() + beg[q];
                    left[l] = cnt[q];
                    off[l] = (uint32_t)(2 * (q / NG) * stride + q % NG);
                    if (steps[r] == 0) empty.push_back((uint16_t)off[l]);
                }
                if (steps[r] == 0) ++me.w;
                for (int k = 0; k < steps[r]; ++k) {
                    int pick[32], banks[4][16] = {}, some = -1;
                    for (int l = 0; l < 32; ++l) {
                        pick[l] = -1;
                        if (left[l] == 0) continue;
                        // of the lane's remaining entries, one whose bank the lanes that load together use least at this step
                        pick[l] = 0;
                        int* use = banks[l / per];
                        for (int j = 1; j < left[l]; ++j)
                            if (use[rem[l][j].ant & (per - 1)] < use[rem[l][pick[l]].ant & (per - 1)]) pick[l] = j;
                        some = rem[l][pick[l]].ant;
                        ++use[some & (per - 1)];
                    }
                    for (int l = 0; l < 32; ++l, ++out) {
                        // past its list a lane gets zero weights and an antenna that another lane reads at this step
                        const uint32_t last = k + 1 == steps[r] ? off[l] << 16 | kGridLast : 0u;
                        if (pick[l] < 0) {
                            key[out] = (uint32_t)some | last;
                            continue;
                        }
                        const Entry& x = rem[l][pick[l]];
                        w[out] = x.w;
                        wim[out] = x.wi;
                        key[out] = (uint32_t)x.ant | last;
                        std::memmove(rem[l] + pick[l], rem[l] + pick[l] + 1, (size_t)(left[l] - pick[l] - 1) * sizeof(Entry));
                        --left[l];
                    }
                }
            }
        }
    }
}

void half256_tables(const std::vector<int>& cptr, const std::vector<int2>& cent, const std::vector<float>& cwim,
                    std::vector<int4>& run, std::vector<float2>& w, std::vector<float2>& wim,
                    std::vector<uint32_t>& key, std::vector<uint16_t>& empty) {
    pair_run_tables(half256::NG, half256::NG, half256::RBS, 16, 16, cptr, cent, cwim, run, w, wim, key, empty);
}

bool half256_fits(int n_ant, size_t smem_optin) {
    return half256::fwd_smem(n_ant) <= smem_optin && half256::bwd_smem(n_ant) <= smem_optin;
}
int half256_row_stride() { return half256::ROWF2; }

cudaError_t launch_half256_fwd(int vdt, const SegList& L, int n_sm, cudaStream_t st) {
    switch (vdt) {
        case 0: return half256::launch_fwd<0>(L, n_sm, st);
        case 1: return half256::launch_fwd<1>(L, n_sm, st);
        case 2: return half256::launch_fwd<2>(L, n_sm, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_half256_bwd(int vdt, const BwdArgs& a, int n_sm, cudaStream_t st) {
    switch (vdt) {
        case 0: return half256::launch_bwd<0>(a, n_sm, st);
        case 1: return half256::launch_bwd<1>(a, n_sm, st);
        case 2: return half256::launch_bwd<2>(a, n_sm, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace epic
