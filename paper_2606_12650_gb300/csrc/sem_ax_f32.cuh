// sem_ax_f32.cuh -- the FP32 line operator of the mixed-precision inner
// solves, one block per few elements, loads straight to registers.
//
// Same map, even-odd products and order of operations as lines_group
// (sem_ax_lines.cuh); y is bit-identical to it.  What differs is how the bytes
// move.  The FP32 operator is bound by HBM: per local node 12 (BF16) or 24
// bytes of factors, x and y, and in an inner CG iteration r, p and d read, p,
// d and w written.  Each thread loads its t line (coalesced over the lines of
// an element) and its nodes' factors itself and nothing waits for a staged
// slab: 64 registers and three padded buffers leave 28 to 32 warps per SM with
// all their loads in flight.  E = 32^3, N = 7, BF16 factors: y = A x 65 -> 58
// us, against 51 us for its bytes at the measured copy rate.
//
// In CG mode the block stores its part of <p, A p> and leaves; pap_sum_kernel
// adds the parts and forms alpha.  A block lives ~4 us here, and a ticket at
// its end (store, fence, atomic, wait) holds its slot ~1.3 us longer: 90 us
// with it, 76 us without (E = 32^3, N = 7, BF16, d not yet updated here), and
// the sum over 16384 parts takes 3 us.
//
// d += alpha p of the previous iteration is applied here (d given), where the old p is
// in registers anyway (+17 us), which leaves the update kernel with r and w
// alone (sem_box.cuh, 72 -> 39 us).
#pragma once

#include "sem_ax_lines.cuh"

namespace sem {

// One node's six factors as stored, and widened to FP32.
template <typename GT>
struct GNode;
template <>
struct GNode<__nv_bfloat16> {
    unsigned w[3];
    __device__ __forceinline__ void load(const __nv_bfloat16 *G, int64_t node) {
        const unsigned *q = reinterpret_cast<const unsigned *>(G + 6 * node);
        w[0] = __ldg(q);
        w[1] = __ldg(q + 1);
        w[2] = __ldg(q + 2);
    }
    __device__ __forceinline__ void get(float (&g)[6]) const {
        const float2 a = bf16x2_to_float2(w[0]), b = bf16x2_to_float2(w[1]), c = bf16x2_to_float2(w[2]);
        g[0] = a.x; g[1] = a.y; g[2] = b.x; g[3] = b.y; g[4] = c.x; g[5] = c.y;
    }
};
template <>
struct GNode<float> {
    float2 w[3];
    __device__ __forceinline__ void load(const float *G, int64_t node) {
        const float2 *q = reinterpret_cast<const float2 *>(G + 6 * node);
        w[0] = __ldg(q);
        w[1] = __ldg(q + 1);
        w[2] = __ldg(q + 2);
    }
    __device__ __forceinline__ void get(float (&g)[6]) const {
        g[0] = w[0].x; g[1] = w[0].y; g[2] = w[1].x; g[3] = w[1].y; g[4] = w[2].x; g[5] = w[2].y;
    }
};

// Per order and factor type: the register limit, and the nodes of a line whose
// factors are loaded before the products (their latency hidden behind them;
// the others are loaded at use, from L2 where the block's prefetch put them).
// Best of 48, 64 and 80 registers with 4 or all nodes, at 1.7e7 nodes.
template <int NQ, typename GT>
struct F32Regs {
    static constexpr bool B16 = sizeof(GT) == 2;
    static constexpr int value = NQ <= 3 ? 48 : (NQ == 10 || (NQ == 9 && !B16) ? 48 : 64);
    static constexpr int early = NQ <= 5 ? NQ : (NQ == 7 || (NQ == 8 && B16) ? NQ : 4);
};

// Buffers padded to rows of odd length: the r lines of a warp start in
// distinct banks (N+1 = 4 and 8 would put 4 or 8 rows in one).
template <int NQ>
struct F32Pad {
    static constexpr int P1 = NQ | 1, P2 = NQ * P1, NPP = NQ * P2;
};
template <int NQ>
__host__ __device__ constexpr size_t f32_smem(int epb) {
    const size_t b = 3 * size_t(epb) * F32Pad<NQ>::NPP * sizeof(float);
    const size_t sum = size_t((epb * NQ * NQ + 31) / 32 * 32) * sizeof(double);   // block_sum_wide's, a double per thread
    return b < sum ? sum : b;
}

// The block's factors towards L2, before its other loads.
template <int NQ, typename GT>
__device__ __forceinline__ void f32_prefetch(const GT *G, int64_t e0, int ne) {
    constexpr int NP = NQ * NQ * NQ;
    if (threadIdx.x == 0) bulk_prefetch_l2(G + 6 * e0 * NP, uint32_t(ne) * NP * 6u * uint32_t(sizeof(GT)));
}

// ne (<= epb) elements from e0.  CG: d += alpha p, p = x + beta p, y = A p, and
// the thread's part of <p, y> in *part; else y = A x.  x, y, p and d are read
// past L1 (the kernel before may have written them while this block already
// waited in pdl_wait).  STATE: beta, alpha and the stop flag come from *st, read
// while the vectors' loads are in flight (false: stopped, nothing written).  In
// a batch the address of the state is itself just loaded, and each such step
// costs 0.7 us of a block's ~5: 256 problems, mixed, 734 -> 615 ms; 32 problems
// 102 -> 92 ms.  A stand-alone solve, whose launches after the stop would read
// its vectors in vain, checks the flag first.
template <int NQ, typename GT, bool CG, bool STATE>
__device__ __forceinline__ bool lines_core_f32(const float *x, float *y, float *p, float *d, const GT *G,
                                               const EoMat<float> &cd, const EoMat<float> &ct, float beta,
                                               float alpha, const CgState *st, int64_t e0, int ne, int epb, float *smem,
                                               float *part) {
    constexpr int NQ2 = NQ * NQ, NP = NQ2 * NQ;
    constexpr int P1 = F32Pad<NQ>::P1, P2 = F32Pad<NQ>::P2, NPP = F32Pad<NQ>::NPP;
    constexpr int GE = F32Regs<NQ, GT>::early;
    const int tid = threadIdx.x;
    const int eb = tid / NQ2, ab = tid - eb * NQ2;
    const int a = ab % NQ, b = ab / NQ;
    const bool act = eb < ne;
    const int64_t nb = (e0 + eb) * NP + ab;   // t line (i, j) = (a, b): first node, stride NQ2
    float *SX = smem + eb * NPP, *SU = SX + epb * NPP, *SV = SU + epb * NPP;
    const int rp = b * P2 + a * P1;   // r line (j, k) = (a, b) of a buffer: first node
    const int cp = b * P2 + a;        // s line (i, k) = (a, b): first node, stride P1
    const int tp = b * P1 + a;        // t line (i, j) = (a, b): first node, stride P2

    float xk[NQ], pv[CG ? NQ : 1], dv[CG ? NQ : 1];
    if (CG && act) {
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
            pv[CG ? k : 0] = __ldcg(p + nb + k * NQ2);
            xk[k] = __ldcg(x + nb + k * NQ2);
            if (d) dv[CG ? k : 0] = __ldcg(d + nb + k * NQ2);
        }
    }
    if (STATE) {
        if (st->done) return false;
        beta = float(st->beta);
        alpha = float(st->alpha);
        f32_prefetch<NQ>(G, e0, ne);
    }
    if (act) {
        if constexpr (CG) {
#pragma unroll
            for (int k = 0; k < NQ; ++k) {
                if (d) d[nb + k * NQ2] = fmaf(alpha, pv[k], dv[k]);
                xk[k] = fmaf(beta, pv[k], xk[k]);
                p[nb + k * NQ2] = xk[k];
            }
        } else {
#pragma unroll
            for (int k = 0; k < NQ; ++k) xk[k] = __ldcg(x + nb + k * NQ2);
        }
#pragma unroll
        for (int k = 0; k < NQ; ++k) SX[k * P2 + tp] = xk[k];
    }
    __syncthreads();

    // gradient lines
    GNode<GT> ge[GE];
    float ut[NQ];
    if (act) {
        float u[NQ], yl[NQ];
#pragma unroll
        for (int l = 0; l < NQ; ++l) u[l] = SX[rp + l];
        eo_apply<NQ, float>(u, yl, cd);
#pragma unroll
        for (int l = 0; l < NQ; ++l) SU[rp + l] = yl[l];
#pragma unroll
        for (int l = 0; l < NQ; ++l) u[l] = SX[cp + l * P1];
        eo_apply<NQ, float>(u, yl, cd);
#pragma unroll
        for (int l = 0; l < NQ; ++l) SV[cp + l * P1] = yl[l];
#pragma unroll
        for (int k = 0; k < GE; ++k) ge[k].load(G, nb + k * NQ2);
        eo_apply<NQ, float>(xk, ut, cd);
    }
    __syncthreads();

    // geometric factors, node by node
    float wt[NQ];
    if (act) {
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
            const int pq = k * P2 + tp;
            const float ur = SU[pq], us = SV[pq];
            float g[6];
            if (k < GE) {
                ge[k < GE ? k : 0].get(g);
            } else {
                GNode<GT> gn;
                gn.load(G, nb + k * NQ2);
                gn.get(g);
            }
            SU[pq] = g[0] * ur + g[1] * us + g[2] * ut[k];
            SV[pq] = g[1] * ur + g[3] * us + g[4] * ut[k];
            wt[k] = g[2] * ur + g[4] * us + g[5] * ut[k];
        }
    }
    __syncthreads();

    // divergence lines (in place: each line has one owner)
    float yt[NQ];
    if (act) {
        float u[NQ], yl[NQ];
#pragma unroll
        for (int l = 0; l < NQ; ++l) u[l] = SU[rp + l];
        eo_apply<NQ, float>(u, yl, ct);
#pragma unroll
        for (int l = 0; l < NQ; ++l) SU[rp + l] = yl[l];
#pragma unroll
        for (int l = 0; l < NQ; ++l) u[l] = SV[cp + l * P1];
        eo_apply<NQ, float>(u, yl, ct);
#pragma unroll
        for (int l = 0; l < NQ; ++l) SV[cp + l * P1] = yl[l];
        eo_apply<NQ, float>(wt, yt, ct);
    }
    __syncthreads();

    float acc = 0.f;
    if (act) {
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
            const int pq = k * P2 + tp;
            const float yv = (SU[pq] + SV[pq]) + yt[k];
            y[nb + k * NQ2] = yv;
            if (CG) acc = fmaf(SX[pq], yv, acc);
        }
    }
    *part = acc;
    return true;
}

template <int NQ, typename GT, bool CG>
__device__ __forceinline__ float lines_group_f32(const float *x, float *y, float *p, float *d, const GT *G,
                                                 const EoMat<float> &cd, const EoMat<float> &ct, float beta,
                                                 float alpha, int64_t e0, int ne, int epb, float *smem) {
    float part;
    lines_core_f32<NQ, GT, CG, false>(x, y, p, d, G, cd, ct, beta, alpha, nullptr, e0, ne, epb, smem, &part);
    return part;
}
template <int NQ, typename GT>
__device__ __forceinline__ bool lines_group_f32_state(const float *x, float *y, float *p, float *d, const GT *G,
                                                      const EoMat<float> &cd, const EoMat<float> &ct, const CgState *st,
                                                      int64_t e0, int ne, int epb, float *smem, float *part) {
    return lines_core_f32<NQ, GT, true, true>(x, y, p, d, G, cd, ct, 0.f, 0.f, st, e0, ne, epb, smem, part);
}

// Blocks that add the n parts of <p, A p>: one up to 2048, else one per 512
// (an FP64 addition of a warp takes 16 cycles: 2048 parts in one block ~0.9
// us, against ~1.3 us more for a second level of blocks).
constexpr int kPapThreads = 256;
__host__ __device__ inline int pap_blocks(int64_t n) {
    if (n <= 2048) return 1;
    const int64_t b = (n + 511) / 512;
    return b < kOneLevel ? int(b) : kOneLevel;
}

// Block b of nb: adds its share of partials[0..n) in a fixed order; the last
// block forms alpha = rho / pap.  The shares' sums go to the slots behind the
// parts (partials + cap), of which there are at least 4096.
__device__ __forceinline__ void pap_sum(double *partials, int64_t cap, int n, int b, int nb, CgState *st) {
    const int per = (n + nb - 1) / nb, first = b * per;
    const double s = block_sum_array(partials + first, max(0, min(per, n - first)));
    double pap = s;
    if (nb > 1) {
        __syncthreads();   // block_sum_array's scratch is free again
        if (!grid_sum(s, partials + cap, cap, &st->ticket_ax, b, nb, &pap)) return;
    }
    if (threadIdx.x == 0) {
        st->pap = pap;
        st->alpha = st->rho / pap;
    }
}

}  // namespace sem
