// sem_ax_fx.cuh -- the FP64 local Poisson operator evaluated in 64-bit
// fixed-point integer arithmetic.
//
// Same map, thread roles and phases as the line kernel (sem_ax_lines.cuh):
// whole r/s/t lines per thread, the even-odd split of D and D^T.  Inputs and
// outputs are FP64 in HBM (x or r, p; y or w; the CG recurrences and
// reductions are untouched).  Inside the kernel an element's values are 64-bit
// integers with one power-of-two scale per element and phase:
//   X = x 2^kx        kx from the largest exponent in the element, |X| < 2^60
//   R = (C . U) / 2^64 for a contraction of U with coefficients C = c 2^kc
// A value v = h 2^32 + l has signed halves (fx_limbs), and a contraction sums
// the exact 64-bit products of halves: the cross terms ch ul + cl uh first
// (from 2^31, so that the cut at 2^32 rounds), their upper half then starts
// the sum of ch uh; cl ul (2^-64 of full scale) is dropped.  Sums of values
// are exact.  The scales of D, of the factors (one exponent per element, kept
// beside them) and of D^T keep every sum below 2^63 for any input
// (fx_coefficients, FxBound).
//
// Every rounding is absolute on the element's scale: together they are below
// 2^-50 of the largest |y| that the element's max |x| and max |G| allow.
// Relative to max |y| itself that depends on how much of those sums cancels.
// Largest error of an element over its max |y|, boxes with sides 1:1:1 to
// 1:30:1000 (the direct FP64 evaluation / pairs of FP32 numbers):
//   random x                  4e-16 at N = 1 .. 4e-15 at N = 9 (2e-16 .. 3e-15 / 1e-14 .. 5e-14)
//   sines over 8 and 32
//   elements a side           N = 3 1e-14, N = 5 1e-13, N = 7 3e-13, N = 9 6e-13
//                             (1e-14, 1e-14, 4e-14, 2e-13 / 4e-13, 2e-12, 4e-12, 7e-12)
//   1 + 1e-6 random           N = 3 3e-10, N = 9 1e-9 (1e-10, 6e-10 / 2e-8, 2e-8)
//   random times 2^-40 .. 1
//   within an element         N = 3 4e-15, N = 9 7e-15 (6e-16, 3e-15 / 2e-14, 2e-14)
//
// Why integers: GB300 runs FP64 at 1/64 of its FP32 rate (DFMA line kernel:
// 1580 us at E = 32^3, N = 7), but a 32 x 32 + 64-bit multiply-add
// (IMAD.WIDE) at half of it: measured 62 per clock and SM, FFMA 119.  A term
// of a contraction costs three of them; in pairs of FP32 numbers (error-free
// sums and products) it took twelve FP32 operations and carried 48 bits.
#pragma once

#include <cmath>

#include "sem_ax_lines.cuh"

namespace sem {

// v = h 2^32 + l, both halves signed.
struct alignas(8) fxl {
    int32_t h, l;
};

constexpr int kFxBits = 60;     // |X| < 2^60
constexpr int kFxGBits = 62;    // |G| < 2^62

// Even-odd coefficients of a centro-antisymmetric matrix (as EoMat), times
// 2^k and rounded to integers.
struct EoMatFX {
    fxl e[25];
    fxl o[30];
    fxl m[5];
    int32_t k, pad;
};

__device__ __forceinline__ fxl fx_limbs(int64_t v) {
    fxl r;
    r.l = int32_t(uint32_t(uint64_t(v)));
    r.h = int32_t(uint64_t(v) >> 32) + int32_t(uint32_t(r.l) >> 31);
    return r;
}

// a b + c in one IMAD.WIDE.  Written as the two halves of a carry chain: the
// assembler rebalances chains of mad.wide into shorter ones joined by 64-bit
// additions (80 of them for the 96 products of an N+1 = 8 line).
__device__ __forceinline__ int64_t fx_mad(int32_t a, int32_t b, int64_t c) {
    int32_t lo = int32_t(uint32_t(uint64_t(c))), hi = int32_t(uint64_t(c) >> 32);
    asm("mad.lo.cc.s32 %0, %2, %3, %0;\n\tmadc.hi.s32 %1, %2, %3, %1;" : "+r"(lo), "+r"(hi) : "r"(a), "r"(b));
    return int64_t((uint64_t(uint32_t(hi)) << 32) | uint32_t(lo));
}

constexpr int64_t kFxHalf = int64_t(1) << 31;
// A sum of cross terms is cut at 2^32, rounded.  Halves go upwards, but away from
// zero at N+1 <= 3, where the coefficients of D are sums of a few powers of two
// and halves frequent: an error of one sign everywhere comes back from a solve
// as A^-1 of it.  At other orders full significands meet a half once in 2^32,
// and away from zero would cost 27 instructions a node (N+1 <= 3: 1 to 3 %).
template <int NQ>
struct FxCut {
    static constexpr int64_t start = NQ <= 3 ? 0 : kFxHalf;   // of the sum
};

__device__ __forceinline__ int64_t fx_cross(fxl c, fxl u, int64_t x) { return fx_mad(c.l, u.h, fx_mad(c.h, u.l, x)); }
__device__ __forceinline__ int64_t fx_upper(int64_t x) { return int64_t(int32_t(uint64_t(x) >> 32)); }

template <int NQ>
__device__ __forceinline__ int64_t fx_cut(int64_t x) {
    return fx_upper(NQ <= 3 ? x + kFxHalf + (x >> 63) : x);
}

// y = M u by the even-odd split (the same sums as eo_apply), st(i, y_i).
template <int NQ, typename Store>
__device__ __forceinline__ void eo_apply_fx(const int64_t (&u)[NQ], const EoMatFX &c, Store st) {
    constexpr int H = NQ / 2;
    constexpr bool ODD = (NQ & 1) != 0;
    fxl ue[H], uo[H], um{};
#pragma unroll
    for (int l = 0; l < H; ++l) {
        ue[l] = fx_limbs(u[l] + u[NQ - 1 - l]);
        uo[l] = fx_limbs(u[l] - u[NQ - 1 - l]);
    }
    if (ODD) um = fx_limbs(u[H]);
#pragma unroll
    for (int i = 0; i < H; ++i) {
        int64_t a = FxCut<NQ>::start, b = a;
#pragma unroll
        for (int l = 0; l < H; ++l) {
            a = fx_cross(c.e[i * H + l], ue[l], a);
            b = fx_cross(c.o[i * H + l], uo[l], b);
        }
        if (ODD) a = fx_cross(c.m[i], um, a);
        a = fx_cut<NQ>(a);
        b = fx_cut<NQ>(b);
#pragma unroll
        for (int l = 0; l < H; ++l) {
            a = fx_mad(c.e[i * H + l].h, ue[l].h, a);
            b = fx_mad(c.o[i * H + l].h, uo[l].h, b);
        }
        if (ODD) a = fx_mad(c.m[i].h, um.h, a);
        st(i, a + b);
        st(NQ - 1 - i, b - a);
    }
    if (ODD) {
        int64_t b = FxCut<NQ>::start;
#pragma unroll
        for (int l = 0; l < H; ++l) b = fx_cross(c.o[H * H + l], uo[l], b);
        b = fx_cut<NQ>(b);
#pragma unroll
        for (int l = 0; l < H; ++l) b = fx_mad(c.o[H * H + l].h, uo[l].h, b);
        st(H, b);
    }
}

// (a . b) / 2^64 of three terms.
template <int NQ>
__device__ __forceinline__ int64_t fx_dot3(fxl a0, fxl a1, fxl a2, fxl b0, fxl b1, fxl b2) {
    int64_t s = fx_cut<NQ>(fx_cross(a2, b2, fx_cross(a1, b1, fx_cross(a0, b0, FxCut<NQ>::start))));
    return fx_mad(a2.h, b2.h, fx_mad(a1.h, b1.h, fx_mad(a0.h, b0.h, s)));
}

// FP64 -> integer: d 2^(kFxBits - 1 - (emax - 1023)) cut to an integer,
// |result| < 2^kFxBits, for an exponent field emax >= d's (>= kFxEmin).
__device__ __forceinline__ int64_t fx_from_double(double d, int emax) {
    const int64_t bits = __double_as_longlong(d);
    const int hi = int(bits >> 32);
    const int e = int((uint32_t(hi) << 1) >> 21);
    const uint64_t m = (uint64_t(uint32_t((hi & 0xfffff) | 0x100000)) << 32) | uint32_t(bits);
    const int64_t v = int64_t((m << (kFxBits - 53)) >> min(emax - e, 63));
    return hi < 0 ? -v : v;
}
// Below this exponent field zero and subnormal inputs (e = 0, whose implicit
// bit fx_from_double adds all the same) would not be shifted out.
constexpr int kFxEmin = 64;

// 2^e as FP64: 0 below and inf above the range of normal numbers.
__device__ __forceinline__ double fx_pow2(int e) {
    const int f = min(max(e + 1023, 0), 2047);
    return __hiloint2double(f << 20, 0);
}

// 1.5 2^52 + v 2^(up - 11) rounded, halves away from zero (|v 2^up| < 2^62):
// A(-x) = -A(x).  Cut instead, or with halves upwards, the error has one sign
// everywhere, and a solve returns A^-1 of it.
__device__ __forceinline__ double fx_top(int64_t v, int up) {
    const int64_t w = int64_t(uint64_t(v) << up);
    return __longlong_as_double(0x4338000000000000ll + ((w + 1024 + (w >> 63)) >> 11));
}

// Shared-memory layout of U, V and X: node (i, j, k) of an element at
// k P2 + j P1 + i, elements NPP apart.  The paddings give the fewest bank
// conflicts of 8-byte values over the row, column and plane steps of a full
// block within 13 % more space (N+1 = 2: 50 %; counted for every padding up to
// +2, +3, +3: N+1 = 8: 3.0 -> 1.5 times the conflict-free wavefronts, N+1 =
// 4: 2.5 -> 1.5, N+1 = 10: 1.48 -> 1.32).
template <int NQ>
struct FxPad {
    static constexpr int P1 = NQ == 8 ? 9 : NQ;
    static constexpr int P2 = NQ == 2 ? 5 : NQ == 4 ? 18 : NQ == 6 ? 38 : NQ == 10 ? 101 : NQ * P1;
    static constexpr int NPP = NQ == 2 ? 12 : NQ == 10 ? 1012 : NQ * P2;
};

// Warps of 32 consecutive threads that the NQ^2 threads of an element can touch.
template <int NQ>
struct FxWarps {
    static constexpr int NQ2 = NQ * NQ;
    static constexpr bool WHOLE = NQ2 % 32 == 0;   // no warp holds threads of two elements
    static constexpr int value = WHOLE ? NQ2 / 32 : (NQ2 + 62) / 32;
};

// Bytes of dynamic shared memory for epb elements: per element and warp one
// 64-bit and one 32-bit word for the reductions, then three regions of 64-bit
// values (which also hold one double per element for the block's final sum).
template <int NQ>
__host__ __device__ constexpr size_t fx_words(int epb) {
    return (size_t(epb) * FxWarps<NQ>::value * 12 + 15) / 16 * 16;
}
template <int NQ>
__host__ __device__ constexpr size_t fx_smem(int epb) {
    return fx_words<NQ>(epb) + 3 * size_t(epb) * FxPad<NQ>::NPP * sizeof(int64_t);
}

// Registers per thread, and the nodes whose factors are loaded ahead of the
// barrier before their use.  The kernel is bound by latency (HBM, and the
// chains of multiply-adds): registers that hold loads in flight compete with
// warps per SM.  Measured over registers x early nodes at ~17 M local nodes
// (CG operator, us): N+1 = 8: 80 x 3 277, 64 x 2 308, 96 x 5 285; N+1 = 9: 80
// x 3 337, 64 x 1 360, 96 x 3 369; N+1 = 10: 96 x 3 397, 64 x 3 491, 112 x 3
// 428; N+1 = 6: 64 x 1 307, 72 x 3 309, 80 x 3 336; N+1 = 4: 64 x 3 255, 72 x
// 3 267; N+1 = 3: 48 x 1 296, 64 x 3 311; N+1 = 2: 40 x 2 326, 64 x 3 397.
template <int NQ>
struct FxRegs {
    static constexpr int value = NQ == 2 ? 40 : NQ == 3 ? 48 : NQ <= 7 ? 64 : NQ <= 9 ? 80 : 96;
    static constexpr int early = NQ == 2 ? 2 : NQ == 4 || NQ >= 8 ? 3 : 1;
};

struct AxFxArgs {
    AxArgs<double, double> a;   // FP64 vectors, state, partials (a.G unused)
    const int4 *G;              // [E][3][NP]: factors (rr, rs), (rt, ss), (st, tt) as halves (h, l, h, l)
    const int32_t *kg;          // [E]: G = g 2^kg
    EoMatFX d;                  // of D   (gradient)
    EoMatFX dt;                 // of D^T (divergence)
    int epb;                    // elements per block
};

// Starts the factors of ne elements from e0, half of the traffic, towards L2
// (before pdl_wait: no kernel of a solve writes them).
template <int NQ>
__device__ __forceinline__ void fx_prefetch(const int4 *G, int64_t e0, int ne) {
    constexpr int NP = NQ * NQ * NQ;
    if (threadIdx.x == 0) bulk_prefetch_l2(G + e0 * (3 * NP), uint32_t(ne) * uint32_t(3 * NP * sizeof(int4)));
}

// The integer factors of one node, from `q` (its element's first plane of
// 16-byte pairs, at the node) with planes NP apart: lanes are consecutive
// nodes, so each load of a warp is one contiguous run.
template <int NP>
__device__ __forceinline__ void load_g6_fx(const int4 *q, int4 (&g)[3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) g[c] = __ldg(q + c * NP);
}

// One group of ne (<= epb) elements starting at element e0, one thread per
// (a, b) of an element.  smem: fx_smem<NQ>(epb) bytes, 16-byte aligned, free
// for all threads.  CG mode: xs += xalpha p_old and p = r + beta p (PRE:
// M^-1 r + beta p) in FP64; *part receives <p, A_local p> of the thread's
// element in the threads (a, b) = (0, 0), 0 in the others (the element's sum
// is formed in integers, so its order does not matter).
//
// Each thread loads and converts its own t line (coalesced: lanes are
// consecutive nodes of a plane), so the vectors need no staging: 2 or 3 loads
// per node are in flight per thread before the first barrier.
template <int NQ, bool CG, bool PRE>
__device__ __forceinline__ void lines_group_fx(const double *x, double *y, double *p, const int4 *G,
                                               const int32_t *kg, const EoMatFX &cd, const EoMatFX &ct, double beta,
                                               double xalpha, double *xs, const double *dinv, int64_t e0, int ne,
                                               int epb, unsigned char *smem, double *part) {
    constexpr int NQ2 = NQ * NQ, NP = NQ2 * NQ;
    constexpr int P1 = FxPad<NQ>::P1, P2 = FxPad<NQ>::P2, NPP = FxPad<NQ>::NPP;
    constexpr bool WHOLE = FxWarps<NQ>::WHOLE;
    constexpr int MW = FxWarps<NQ>::value;
    constexpr int GE = FxRegs<NQ>::early;
    constexpr bool POW2 = NQ2 < 32 && (NQ2 & (NQ2 - 1)) == 0;   // elements are aligned runs of lanes
    int64_t *dots = reinterpret_cast<int64_t *>(smem);
    int *emx = reinterpret_cast<int *>(dots + epb * MW);
    int64_t *reg = reinterpret_cast<int64_t *>(smem + fx_words<NQ>(epb));
    const int tid = threadIdx.x;
    const int eb = tid / NQ2;
    const int ab = tid - eb * NQ2;
    const int a = ab % NQ, b = ab / NQ;
    const bool act = eb < ne;
    const int64_t nb = (e0 + eb) * NP + ab;     // the thread's t line: nb + k NQ2
    // the lanes of this warp in the thread's element (a run of lanes) and the
    // first of them; the warp's word among the element's; their number
    auto lanes_of = [&](int &first) -> uint32_t {
        if (WHOLE) {
            first = 0;
            return 0xffffffffu;
        }
        const int w0 = tid & ~31;
        first = max(eb * NQ2 - w0, 0);
        const int end = min((eb + 1) * NQ2 - w0, 32);
        return (end >= 32 ? 0xffffffffu : (1u << end) - 1u) & ~((1u << first) - 1u);
    };
    auto word_of = [&]() { return WHOLE ? tid >> 5 : eb * MW + (tid >> 5) - (eb * NQ2 >> 5); };
    auto words = [&]() { return WHOLE ? MW : (((eb + 1) * NQ2 - 1) >> 5) - (eb * NQ2 >> 5) + 1; };

    // ---- (0) the thread's t line, and the element's largest exponent
    double v[NQ];
    int kge = 0;
    uint32_t mx = 0;
    if (act) {
        kge = __ldg(kg + e0 + eb);
        if (CG) {
            double pv[NQ];
#pragma unroll
            for (int k = 0; k < NQ; ++k) {
                pv[k] = __ldcg(p + nb + k * NQ2);   // from L2, see vload_cg in sem_box.cuh
                v[k] = __ldcg(x + nb + k * NQ2);
                if (PRE) v[k] *= __ldg(dinv + nb + k * NQ2);
            }
            if (xs) {
                double xv[NQ];
#pragma unroll
                for (int k = 0; k < NQ; ++k) xv[k] = __ldcg(xs + nb + k * NQ2);
#pragma unroll
                for (int k = 0; k < NQ; ++k) xs[nb + k * NQ2] = fma(xalpha, pv[k], xv[k]);
            }
#pragma unroll
            for (int k = 0; k < NQ; ++k) {
                v[k] = fma(beta, pv[k], v[k]);
                p[nb + k * NQ2] = v[k];
            }
        } else {
#pragma unroll
            for (int k = 0; k < NQ; ++k) v[k] = __ldcg(x + nb + k * NQ2);
        }
#pragma unroll
        for (int k = 0; k < NQ; ++k) mx = max(mx, uint32_t(__double2hiint(v[k])) & 0x7fffffffu);
    }
    {
        int first;
        const uint32_t lanes = lanes_of(first);
        if (POW2) {
#pragma unroll
            for (int o = NQ2 / 2; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        } else {
            mx = __reduce_max_sync(lanes, mx);
        }
        if (act && (tid & 31) == first) emx[word_of()] = int(mx);
    }
    __syncthreads();
    int64_t *SX = reg + eb * NPP;
    int64_t *SU = SX + epb * NPP;
    int64_t *SV = SU + epb * NPP;
    const int rp = b * P2 + a * P1;    // r line (j, k) = (a, b)
    const int cp = b * P2 + a;         // s line (i, k) = (a, b), stride P1
    const int tp = b * P1 + a;         // t line (i, j) = (a, b), stride P2
    int emax = 0;
    int64_t X[NQ];
    if (act) {
        int em = kFxEmin << 20;
#pragma unroll
        for (int j = 0; j < MW; ++j)
            if (j < words()) em = max(em, emx[eb * MW + j]);
        emax = em >> 20;
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
            X[k] = fx_from_double(v[k], emax);
            SX[k * P2 + tp] = X[k];
        }
    }
    __syncthreads();

    // ---- (1) gradient lines; the r and s lines share one copy of the code.
    // The factors of the first nodes start into registers at the end.
    int64_t ut[NQ];
    int4 ge[GE][3];
    const int4 *Ge = G + (e0 + eb) * (3 * NP) + ab;
    if (act) {
        eo_apply_fx<NQ>(X, cd, [&](int i, int64_t w) { ut[i] = w; });
#pragma unroll 1
        for (int d = 0; d < 2; ++d) {
            const int64_t *src = SX + (d ? cp : rp);
            int64_t *dst = d ? SV + cp : SU + rp;
            const int st = d ? P1 : 1;
            int64_t u[NQ];
#pragma unroll
            for (int l = 0; l < NQ; ++l) u[l] = src[l * st];
            eo_apply_fx<NQ>(u, cd, [&](int i, int64_t w) { dst[i * st] = w; });
        }
#pragma unroll
        for (int k = 0; k < GE; ++k) load_g6_fx<NP>(Ge + k * NQ2, ge[k]);
    }
    __syncthreads();

    // ---- (2) geometric factors, node by node
    int64_t wt[NQ];
    if (act) {
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
            const int pq = k * P2 + tp;
            int4 g[3];
            if (k < GE) {
#pragma unroll
                for (int c = 0; c < 3; ++c) g[c] = ge[k < GE ? k : 0][c];
            } else {
                load_g6_fx<NP>(Ge + k * NQ2, g);
            }
            const fxl ur = fx_limbs(SU[pq]), us = fx_limbs(SV[pq]), uv = fx_limbs(ut[k]);
            const fxl rr{g[0].x, g[0].y}, rs{g[0].z, g[0].w}, rt{g[1].x, g[1].y}, ss{g[1].z, g[1].w},
                s_t{g[2].x, g[2].y}, tt{g[2].z, g[2].w};
            SU[pq] = fx_dot3<NQ>(rr, rs, rt, ur, us, uv);
            SV[pq] = fx_dot3<NQ>(rs, ss, s_t, ur, us, uv);
            wt[k] = fx_dot3<NQ>(rt, s_t, tt, ur, us, uv);
        }
    }
    __syncthreads();

    // ---- (3) divergence lines (in place: each line has one owner)
    int64_t yt[NQ];
    if (act) {
        eo_apply_fx<NQ>(wt, ct, [&](int i, int64_t w) { yt[i] = w; });
#pragma unroll 1
        for (int d = 0; d < 2; ++d) {
            int64_t *line = d ? SV + cp : SU + rp;
            const int st = d ? P1 : 1;
            int64_t u[NQ];
#pragma unroll
            for (int l = 0; l < NQ; ++l) u[l] = line[l * st];
            eo_apply_fx<NQ>(u, ct, [&](int i, int64_t w) { line[i * st] = w; });
        }
    }
    __syncthreads();

    // ---- (4) sum of the three directions and <p, y>; y = Y 2^q, shifted up by
    // the thread's common headroom and rounded to 51 bits for FP64 (one FMA)
    const int q = emax - (kFxBits - 53 + 1075) - cd.k - ct.k + 192 - kge;
    int64_t dot = 0;
    if (act) {
        int64_t acc = kFxHalf;
        uint32_t top = 0;
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
            const int pq = k * P2 + tp;
            yt[k] += SU[pq] + SV[pq];
            const int h = int(yt[k] >> 32);
            top |= uint32_t(h ^ (h >> 31));
            if (CG) {
                const fxl yl = fx_limbs(yt[k]), xl = fx_limbs(SX[pq]);
                acc = fx_cross(xl, yl, acc);
                dot = fx_mad(xl.h, yl.h, dot);
                if (NQ == 10 && k == 4) {   // ten nodes' cross terms could pass 2^63
                    dot += fx_upper(acc);
                    acc = kFxHalf;
                }
            }
        }
        dot += fx_upper(acc);
        const int up = max(__clz(int(top)) - 2, 0);
        // a NaN or an infinity in the element makes all of its y NaN
        const double f = emax == 2047 ? __hiloint2double(0x7ff80000, 0) : fx_pow2(q - up + 11);
        const double f0 = -0x1.8p52 * f;
#pragma unroll
        for (int k = 0; k < NQ; ++k)
            y[nb + k * NQ2] = fma(fx_top(yt[k], up), f, f0);
    }
    if (CG) {
        // the element's sum of X Y / 2^64: per warp by shuffles or as three
        // 32-bit sums (each of 32 values below 2^22, the last one signed), then
        // over the warps
        int64_t t = act ? dot : 0;
        int first;
        const uint32_t lanes = lanes_of(first);
        if (POW2) {
#pragma unroll
            for (int o = NQ2 / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        } else {
            const uint32_t s0 = __reduce_add_sync(lanes, uint32_t(t) & 0x3fffffu);
            const uint32_t s1 = __reduce_add_sync(lanes, uint32_t(uint64_t(t) >> 22) & 0x3fffffu);
            const int32_t s2 = __reduce_add_sync(lanes, int32_t(t >> 44));
            t = int64_t(s0) + (int64_t(s1) << 22) + (int64_t(s2) << 44);
        }
        if (act && (tid & 31) == first) dots[word_of()] = t;
        __syncthreads();
        double pt = 0.0;
        if (act && ab == 0) {
            int64_t sum = 0;
            for (int j = 0; j < words(); ++j) sum += dots[eb * MW + j];
            pt = double(sum) *
                 (emax == 2047 ? __hiloint2double(0x7ff80000, 0) : fx_pow2(q + 64 + emax - (kFxBits - 53 + 1075)));
        }
        *part = pt;
    }
}

// Block b of nb after lines_group_fx: the block's <p, A_local p>, and in the
// last block alpha = rho / <p, A p>.
template <int NQ>
__device__ __forceinline__ void fx_publish(double part, unsigned char *smem, int epb, double *partials, int64_t cap,
                                           CgState *st, int b, int nb) {
    double bs = part;
    if (epb > 1) {
        // the regions are free: every thread passed lines_group_fx's last barrier after its reads
        double *sums = reinterpret_cast<double *>(smem + fx_words<NQ>(epb));
        const int eb = threadIdx.x / (NQ * NQ);
        if (int(threadIdx.x) == eb * NQ * NQ && eb < epb) sums[eb] = part;
        __syncthreads();
        bs = 0.0;
        if (threadIdx.x < 32) {
            for (int k = threadIdx.x; k < epb; k += 32) bs += sums[k];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (o < epb) bs += __shfl_down_sync(0xffffffffu, bs, o);
        }
    }
    double pap;
    if (grid_sum(bs, partials, cap, &st->ticket_ax, b, nb, &pap) && threadIdx.x == 0) {
        st->pap = pap;
        st->alpha = st->rho / pap;
    }
}

template <int NQ, bool CG, bool PRE>
__global__ void __maxnreg__(FxRegs<NQ>::value) ax_fx_kernel(const __grid_constant__ AxFxArgs P) {
    extern __shared__ __align__(16) unsigned char smem[];
    const AxArgs<double, double> &A = P.a;
    const int64_t e0 = int64_t(blockIdx.x) * P.epb;
    const int ne = int(min(int64_t(P.epb), A.E - e0));
    if (!CG) fx_prefetch<NQ>(P.G, e0, ne);
    pdl_wait();
    if (CG && A.st->done) return;  // solve finished: the rest of the graph is a no-op
    if (CG) fx_prefetch<NQ>(P.G, e0, ne);
    const double beta = CG ? A.st->beta : 0.0;
    // read before this launch's last block replaces it; only with a deferred x update
    const double xalpha = (CG && A.xs) ? A.st->alpha : 0.0;
    double part = 0.0;
    lines_group_fx<NQ, CG, PRE>(A.x, A.y, A.p, P.G, P.kg, P.d, P.dt, beta, xalpha, CG ? A.xs : nullptr, A.dinv, e0, ne,
                                P.epb, smem, &part);
    if (CG) fx_publish<NQ>(part, smem, P.epb, A.partials, A.cap, A.st, int(blockIdx.x), int(gridDim.x));
}

// Host: the even-odd halves of M (row-major nq x nq) times 2^k, rounded to
// integers, for inputs |u| < ubound (integers): the largest k for which
//   - every coefficient's upper half fits 32 bits, and
//   - the cross terms of any row, sum |ch| 2^31 + sum |uh| 2^31, stay below 2^63
// (u_e, u_o < 2 ubound).  Both bound the sum of the upper products too.
// *ybound: the bound of |M u| / 2^64 * 2^k.
inline EoMatFX eo_coefficients_fx(const double *M, int nq, double ubound, double *ybound) {
    const int N = nq - 1, H = nq / 2;
    const bool odd = (nq & 1) != 0;
    auto e = [&](int i, int l) { return 0.5 * (M[i * nq + l] + M[i * nq + N - l]); };
    auto o = [&](int i, int l) { return 0.5 * (M[i * nq + l] - M[i * nq + N - l]); };
    double big = 0.0, row = 0.0, full = 0.0;
    for (int i = 0; i < H + (odd ? 1 : 0); ++i) {
        double se = 0.0, so = 0.0, sf = 0.0;
        for (int l = 0; l < H; ++l) {
            if (i < H) se += std::fabs(e(i, l));
            so += std::fabs(o(i, l));
            if (i < H) big = std::max(big, std::fabs(e(i, l)));
            big = std::max(big, std::fabs(o(i, l)));
        }
        if (odd && i < H) {
            se += std::fabs(M[i * nq + H]);
            big = std::max(big, std::fabs(M[i * nq + H]));
        }
        for (int l = 0; l < nq; ++l) sf += std::fabs(M[i * nq + l]);
        row = std::max(row, std::max(se, so));
        full = std::max(full, sf);
    }
    const double two32 = 4294967296.0;
    const double uh = (2.0 * H * ubound + (odd ? ubound : 0.0)) / two32 + 2 * H + 2;
    int k = 0;
    while (std::ldexp(big, k + 1) < std::ldexp(1.0, 63) - two32 &&
           (std::ldexp(row, k + 1) / two32 + uh) * std::ldexp(1.0, 31) < std::ldexp(1.0, 63))
        ++k;
    EoMatFX c{};
    c.k = k;
    auto fix = [k](double d) {
        const int64_t v = std::llrint(std::ldexp(d, k));
        fxl r;
        r.l = int32_t(uint32_t(uint64_t(v)));
        r.h = int32_t((v - int64_t(r.l)) >> 32);
        return r;
    };
    for (int i = 0; i < H; ++i)
        for (int l = 0; l < H; ++l) {
            c.e[i * H + l] = fix(e(i, l));
            c.o[i * H + l] = fix(o(i, l));
        }
    if (odd) {
        for (int l = 0; l < H; ++l) c.o[H * H + l] = fix(o(H, l));
        for (int i = 0; i < H; ++i) c.m[i] = fix(M[i * nq + H]);
    }
    *ybound = std::ldexp(full, k - 64) * ubound;
    return c;
}

// A problem's matrices, made once beside its factors (~2 us on the host, of a
// launch's 8).
struct FxConsts {
    EoMatFX d, dt;
};

// What bounds an element's sum of |X Y| / 2^64: with |X| < 2^60, the row sums
// rows[i] of |D| and G = g 2^61 (|g| < 2),
//   2^(k + kt - 75) S,  S = sum over nodes and a, b of rows_a |g_ab| rows_b.
struct FxBound {
    float rows[kMaxQ];
    float limit;      // of S, for a sum below 2^62
};

inline FxBound fx_bound(const double *D, int nq, int k, int kt) {
    FxBound b{};
    for (int i = 0; i < nq; ++i) {
        double s = 0.0;
        for (int l = 0; l < nq; ++l) s += std::fabs(D[i * nq + l]);
        b.rows[i] = float(s);
    }
    b.limit = float(std::ldexp(0.99, 62 + 75 - k - kt));
    return b;
}

// Host: both matrices of an order.  |X| < 2^kFxBits, |W| <= 3 2^kFxGBits |D X|.
inline void fx_coefficients(const double *D, int nq, EoMatFX *d, EoMatFX *dt) {
    double Dt[kMaxQ * kMaxQ], b1, b2;
    for (int i = 0; i < nq; ++i)
        for (int l = 0; l < nq; ++l) Dt[i * nq + l] = D[l * nq + i];
    *d = eo_coefficients_fx(D, nq, std::ldexp(1.0, kFxBits), &b1);
    *dt = eo_coefficients_fx(Dt, nq, std::ldexp(3.0, kFxGBits - 64) * b1, &b2);
}

}  // namespace sem
