// sem_cg_small.cu -- FP64 CG to a tolerance and Jacobi-PCG of problems whose
// elements all fit the GPU at once: one cooperative kernel runs the whole solve,
// a block per element.  An iteration of CG, graph of two launches -> this kernel, in us: N
// = 7: E = 64 17.4 -> 13.0, 150 19.7 -> 14.1, 448 22.8 -> 19.6; N = 5: 384
// 20.1 -> 14.3; N = 9: 64 21.5 -> 16.8; N = 3: 343 15.2 -> 11.9.
//
// The two launches of an iteration (sem_cg.cu) are bound by latency when a
// problem gives an SM an element or less: E = 64, N = 7 takes 18 us an
// iteration, of which the bytes would take 0.5.  Here a block keeps its
// element's x, r and p in registers for the whole solve, and per iteration
// exchanges only what crosses elements: w at the nodes on element faces, and
// the block's parts of <p, A p> and <r, r>.
//
// Exchange.  A block writes its face nodes' w, then its part into its slot, as
// two 64-bit words each holding half of the value and the iteration number, so
// that a word is never seen half written and needs no separate flag.  Every
// block polls all slots until they carry the iteration's number and adds them
// in the same order, so all blocks hold the same bits of alpha, beta and the
// stop flag and nothing has to be sent back.  A block leaves an exchange only
// when every block has entered it, so the other exchange's slots are free
// again; w alternates between two buffers (the second one is p's, which is in
// registers meanwhile), so that a block's reads of one are ordered before its
// next writes to it by the fences of the exchange in between, and only the
// exchange after w needs fences.  The waits are bounded (status word); the
// cooperative launch makes all blocks resident, and a launch runs a bounded
// number of iterations.  It starts when all its blocks fit, so such a solve waits
// for other streams' kernels to leave room instead of running beside them.
//
// Threads.  Three per (a, b) of an element, one for each direction: thread (d,
// a, b) takes the line (a, b) of direction d in the contractions, and the
// nodes (a, b, d + 3 s) elsewhere, so that an element's contraction is one line
// deep instead of three.  The arithmetic is the fixed-point operator's
// (sem_ax_fx.cuh).  At full occupancy this split is slower (E = 32^3, N = 7:
// 356 against 279 us: the t line goes through shared memory too), which is why
// larger problems do not use it.
#include <cuda_runtime.h>

#include <algorithm>

#include "sem_ax_fx.cuh"
#include "sem_box.cuh"
#include "sem_device.cuh"
#include "sem_internal.h"

namespace sem {
namespace {

struct SmallArgs {
    double *x, *r, *p, *w;
    const double *dinv;
    const int4 *G;
    const int32_t *kg;
    EoMatFX d, dt;
    int nx, ny, nz;
    int iters;              // iterations of this launch at most
    CgState *st;
    uint64_t *slots;        // zero at the launch: 2 words per block and group, then 2 or 4
    int32_t *status;
    uint64_t limit_ns;      // of a wait
};

template <int NQ>
struct SmallShape {
    static constexpr int NQ2 = NQ * NQ, NT = 3 * NQ2;
    static constexpr int T = (NT + 31) / 32 * 32, W = T / 32;
    static constexpr int KS = (NQ + 2) / 3;
    static constexpr int regs = NQ <= 5 ? 64 : NQ <= 9 ? 80 : 96;
    static constexpr size_t smem = 4 * size_t(FxPad<NQ>::NPP) * sizeof(int64_t);
};

__device__ __forceinline__ void put_word(uint64_t *q, uint32_t value, uint32_t epoch) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(q), "l"((uint64_t(epoch) << 32) | value) : "memory");
}
__device__ __forceinline__ void put_value(uint64_t *q, double v, uint32_t epoch) {
    put_word(q, uint32_t(__double2loint(v)), epoch);
    put_word(q + 1, uint32_t(__double2hiint(v)), epoch);
}
__device__ __forceinline__ void get_words(const uint64_t *q, uint64_t &v0, uint64_t &v1) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v0), "=l"(v1) : "l"(q) : "memory");
}

constexpr uint64_t kExchangeLimitNs = 4000000000ull;

// This thread's share (slots tid, tid + blockDim, ...) of the sums of the NV
// values of n slots, once they carry `epoch`; FENCE: what their writers wrote
// before is then visible after the block's next barrier.  false: the wait ran
// out.
template <int NV, bool FENCE>
__device__ __forceinline__ bool get_share(const uint64_t *slots, int n, uint32_t epoch, double (&sum)[NV],
                                          uint64_t limit_ns) {
#pragma unroll
    for (int c = 0; c < NV; ++c) sum[c] = 0.0;
    for (int q = threadIdx.x; q < n; q += blockDim.x) {
        const uint64_t *s = slots + size_t(2 * NV) * q;
        uint64_t v[2 * NV], t0 = 0;
        for (unsigned it = 0;; ++it) {
            bool all = true;
#pragma unroll
            for (int c = 0; c < 2 * NV; c += 2) {
                get_words(s + c, v[c], v[c + 1]);
                all &= uint32_t(v[c] >> 32) == epoch && uint32_t(v[c + 1] >> 32) == epoch;
            }
            if (all) break;
            if (it == 0) {
                t0 = global_ns();
            } else if ((it & 63u) == 0 && global_ns() - t0 > limit_ns) {
                return false;
            }
        }
#pragma unroll
        for (int c = 0; c < NV; ++c)
            sum[c] += __hiloint2double(int(uint32_t(v[2 * c + 1])), int(uint32_t(v[2 * c])));
    }
    if (FENCE && threadIdx.x < n) __threadfence();
    return true;
}

// Exchange of NV values per block (lane 0 of warp 0 holds this block's): the
// block's slot, then, beyond kDirect blocks, one slot per group of 32 blocks,
// which the group's first block fills (every block polling every slot costs
// 6 us more an iteration at 512 blocks, 0.8 at 64, and 0.6 less at 32).  This thread's share of the sums goes to
// `share`, of *n slots in all.
constexpr int kDirect = 32;
template <int NV, bool FENCE>
__device__ __forceinline__ bool exchange(uint64_t *slots, int nb, int e, uint32_t epoch, const double (&mine)[NV],
                                         double (&share)[NV], int *n, uint64_t limit_ns) {
    if (threadIdx.x == 0) {
        if (FENCE) __threadfence();   // the block's writes and reads of w before its slot
#pragma unroll
        for (int c = 0; c < NV; ++c) put_value(slots + 2 * (size_t(NV) * e + c), mine[c], epoch);
    }
    *n = nb;
    if (nb <= kDirect) return get_share<NV, FENCE>(slots, nb, epoch, share, limit_ns);
    uint64_t *groups = slots + size_t(2 * NV) * nb;
    *n = (nb + 31) / 32;
    bool ok = true;
    if (e % 32 == 0 && threadIdx.x < 32) {
        double v[NV];
        ok = get_share<NV, FENCE>(slots + size_t(2 * NV) * e, min(32, nb - e), epoch, v, limit_ns);
        ok = __all_sync(0xffffffffu, ok);
        // orders every lane's reads (and fence) before lane 0's store below: votes
        // and shuffles do not order memory between lanes
        __syncwarp();
#pragma unroll
        for (int c = 0; c < NV; ++c) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v[c] += __shfl_down_sync(0xffffffffu, v[c], o);
        }
        if (ok && threadIdx.x == 0) {
            if (FENCE) __threadfence();
#pragma unroll
            for (int c = 0; c < NV; ++c) put_value(groups + 2 * (size_t(NV) * (e / 32) + c), v[c], epoch);
        }
    }
    return get_share<NV, FENCE>(groups, *n, epoch, share, limit_ns) && ok;
}

// Sum of v over the first n threads, in warp 0 (all lanes take part, the
// result is lane 0's); after a barrier that orders the threads' stores of v.
__device__ __forceinline__ double warp0_sum(const double *v, int n) {
    double s = 0.0;
    for (int q = threadIdx.x; q < n; q += 32) s += v[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    return s;
}

template <int NQ, bool PRE>
__global__ void __maxnreg__(SmallShape<NQ>::regs) cg_small_kernel(const __grid_constant__ SmallArgs A) {
    using S = SmallShape<NQ>;
    constexpr int NQ2 = S::NQ2, NP = NQ2 * NQ, NT = S::NT, KS = S::KS, W = S::W, N = NQ - 1;
    constexpr int P1 = FxPad<NQ>::P1, P2 = FxPad<NQ>::P2, RG = FxPad<NQ>::NPP;
    constexpr int NV2 = PRE ? 2 : 1;
    extern __shared__ __align__(16) int64_t SX[];   // X, then the lines of the three directions, RG apart
    __shared__ int s_max[W];
    __shared__ int64_t s_dot[W];
    __shared__ double s_red[NV2][S::T];
    __shared__ double s_bc[2];
    __shared__ int s_stop;

    CgState *st = A.st;
    if (st->done) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool act = tid < NT;
    const int d = tid / NQ2, ab = tid - d * NQ2;
    const int b = ab / NQ, a = ab - b * NQ;
    const int e = blockIdx.x, nb = gridDim.x;
    const int ex = e % A.nx, ey = e / A.nx % A.ny, ez = e / A.nx / A.ny;
    const int l0 = e * NP + tid;                     // node s: l0 + s NT, (i, j, k) = (a, b, d + 3 s)
    uint64_t *slots1 = A.slots, *slots2 = A.slots + 2 * size_t(nb + (nb + 31) / 32);

    // the neighbour element's copy of a node on a face: -1, 0, 1 per direction
    const int sx = a == 0 && ex > 0 ? -1 : (a == N && ex < A.nx - 1 ? 1 : 0);
    const int sy = b == 0 && ey > 0 ? -1 : (b == N && ey < A.ny - 1 ? 1 : 0);
    const bool mxy = (a == 0 && ex == 0) || (a == N && ex == A.nx - 1) || (b == 0 && ey == 0) ||
                     (b == N && ey == A.ny - 1);
    const int ox = sx * (NP - N), oy = sy * (A.nx * NP - N * NQ), oz1 = A.nx * A.ny * NP - N * NQ2;
    auto sz_of = [&](int s) {
        const int k = d + 3 * s;
        return k == 0 && ez > 0 ? -1 : (k == N && ez < A.nz - 1 ? 1 : 0);
    };
    auto masked = [&](int s) {
        const int k = d + 3 * s;
        return mxy || (k == 0 && ez == 0) || (k == N && ez == A.nz - 1);
    };

    double x[KS], r[KS], p[KS], wv[KS], dv[PRE ? KS : 1];
    int kge = 0;
#pragma unroll
    for (int s = 0; s < KS; ++s) {
        x[s] = r[s] = p[s] = wv[s] = 0.0;
        if (PRE) dv[PRE ? s : 0] = 0.0;
        if (act && d + 3 * s < NQ) {
            x[s] = A.x[l0 + s * NT];
            r[s] = A.r[l0 + s * NT];
            p[s] = A.p[l0 + s * NT];
            if (PRE) dv[PRE ? s : 0] = A.dinv[l0 + s * NT];
        }
    }
    if (act) kge = A.kg[e];
    double beta = st->beta, alpha = 0.0;
    // the recurrence's scalars live in thread 0
    double rho = st->rho, pap = 0.0, rr = 0.0;
    const double ref = PRE ? st->bb : st->rho0;
    // the stop test sqrt(rr / ref) <= tol as rr / ref <= t2, t2 the largest
    // number whose (correctly rounded) root is at most tol: no root in the loop
    const double tol = st->tol;
    double t2 = -1.0;
    if (tol > 0.0) {
        t2 = tol * tol;
        while (sqrt(t2) > tol) t2 = __longlong_as_double(__double_as_longlong(t2) - 1);
        while (t2 < 1e300 && sqrt(__longlong_as_double(__double_as_longlong(t2) + 1)) <= tol)
            t2 = __longlong_as_double(__double_as_longlong(t2) + 1);
    }
    double *hist = st->hist;
    int iter = st->iter;
    const int iter0 = iter, maxit = st->maxit;

    const int stride = d == 0 ? 1 : (d == 1 ? P1 : P2);
    const int line0 = d == 0 ? b * P2 + a * P1 : (d == 1 ? b * P2 + a : b * P1 + a);
    const int tp = d * P2 + b * P1 + a;              // node s: tp + 3 s P2
    int64_t *line = SX + (d + 1) * RG + line0;
    const int4 *Ge = A.G + size_t(e) * (3 * NP) + tid;

    int n = 1;
    for (;; ++n) {
        double *w = n & 1 ? A.w : A.p;
        // ---- p = z + beta p, in integers of the element's scale
        uint32_t mx = 0;
#pragma unroll
        for (int s = 0; s < KS; ++s) {
            p[s] = fma(beta, p[s], PRE ? dv[PRE ? s : 0] * r[s] : r[s]);
            mx = max(mx, uint32_t(__double2hiint(p[s])) & 0x7fffffffu);
        }
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0) s_max[warp] = int(mx);
        __syncthreads();
        int em = kFxEmin << 20;
#pragma unroll
        for (int q = 0; q < W; ++q) em = max(em, s_max[q]);
        const int emax = em >> 20;
        if (act) {
#pragma unroll
            for (int s = 0; s < KS; ++s)
                if (d + 3 * s < NQ) SX[tp + 3 * s * P2] = fx_from_double(p[s], emax);
        }
        __syncthreads();
        // ---- gradient: this thread's line
        if (act) {
            int64_t u[NQ];
            const int64_t *src = SX + line0;
#pragma unroll
            for (int l = 0; l < NQ; ++l) u[l] = src[l * stride];
            eo_apply_fx<NQ>(u, A.d, [&](int i, int64_t v) { line[i * stride] = v; });
        }
        __syncthreads();
        // ---- geometric factors
        if (act) {
#pragma unroll
            for (int s = 0; s < KS; ++s)
                if (d + 3 * s < NQ) {
                    int4 g[3];
                    load_g6_fx<NP>(Ge + s * NT, g);
                    int64_t *q = SX + RG + tp + 3 * s * P2;
                    const fxl ur = fx_limbs(q[0]), us = fx_limbs(q[RG]), ut = fx_limbs(q[2 * RG]);
                    const fxl grr{g[0].x, g[0].y}, grs{g[0].z, g[0].w}, grt{g[1].x, g[1].y}, gss{g[1].z, g[1].w},
                        gst{g[2].x, g[2].y}, gtt{g[2].z, g[2].w};
                    q[0] = fx_dot3<NQ>(grr, grs, grt, ur, us, ut);
                    q[RG] = fx_dot3<NQ>(grs, gss, gst, ur, us, ut);
                    q[2 * RG] = fx_dot3<NQ>(grt, gst, gtt, ur, us, ut);
                }
        }
        __syncthreads();
        // ---- divergence, in place
        if (act) {
            int64_t u[NQ];
#pragma unroll
            for (int l = 0; l < NQ; ++l) u[l] = line[l * stride];
            eo_apply_fx<NQ>(u, A.dt, [&](int i, int64_t v) { line[i * stride] = v; });
        }
        __syncthreads();
        // ---- w = A p; face nodes to memory; the element's part of <p, w>
        const int q0 = emax - (kFxBits - 53 + 1075) - A.d.k - A.dt.k + 192 - kge;
        int64_t dot = 0;
        if (act) {
            int64_t Y[KS], acc = kFxHalf;
            uint32_t top = 0;
#pragma unroll
            for (int s = 0; s < KS; ++s)
                if (d + 3 * s < NQ) {
                    const int64_t *q = SX + tp + 3 * s * P2;
                    Y[s] = q[RG] + q[2 * RG] + q[3 * RG];
                    const int h = int(Y[s] >> 32);
                    top |= uint32_t(h ^ (h >> 31));
                    const fxl yl = fx_limbs(Y[s]), xl = fx_limbs(q[0]);
                    acc = fx_cross(xl, yl, acc);
                    dot = fx_mad(xl.h, yl.h, dot);
                }
            dot += fx_upper(acc);
            const int up = max(__clz(int(top)) - 2, 0);
            const double f = emax == 2047 ? __hiloint2double(0x7ff80000, 0) : fx_pow2(q0 - up + 11);
            const double f0 = -0x1.8p52 * f;
#pragma unroll
            for (int s = 0; s < KS; ++s)
                if (d + 3 * s < NQ) {
                    wv[s] = fma(fx_top(Y[s], up), f, f0);
                    if (sx || sy || sz_of(s)) __stcg(w + l0 + s * NT, wv[s]);
                }
        }
        {
            const uint32_t t0 = __reduce_add_sync(0xffffffffu, uint32_t(dot) & 0x3fffffu);
            const uint32_t t1 = __reduce_add_sync(0xffffffffu, uint32_t(uint64_t(dot) >> 22) & 0x3fffffu);
            const int32_t t2 = __reduce_add_sync(0xffffffffu, int32_t(dot >> 44));
            if (lane == 0) s_dot[warp] = int64_t(t0) + (int64_t(t1) << 22) + (int64_t(t2) << 44);
        }
        __syncthreads();
        double part[1] = {0.0};
        if (tid == 0) {
            int64_t sum = 0;
#pragma unroll
            for (int q = 0; q < W; ++q) sum += s_dot[q];
            part[0] = double(sum) * (emax == 2047 ? __hiloint2double(0x7ff80000, 0)
                                                  : fx_pow2(q0 + 64 + emax - (kFxBits - 53 + 1075)));
        }
        // ---- first exchange: every block's part, and its w
        double share1[1];
        int ns;
        const bool ok1 = exchange<1, true>(slots1, nb, e, uint32_t(n), part, share1, &ns, A.limit_ns);
        s_red[0][tid] = share1[0];
        if (__syncthreads_or(!ok1)) {
            if (tid == 0) atomicExch(A.status, int32_t(kStatusExchangeTimeout));
            return;
        }
        double c[KS];
        if (act) {
            // the copies, added pairwise by direction: the sum is the same in
            // every copy, whichever of the two is its own
#pragma unroll
            for (int s = 0; s < KS; ++s)
                if (d + 3 * s < NQ) {
                    const double *q = w + l0 + s * NT;
                    const int sz = sz_of(s), oz = sz * oz1;
                    const double wx = sx ? __ldcg(q + ox) : 0.0;
                    double wy = 0.0, wxy = 0.0, wz = 0.0, wxz = 0.0, wyz = 0.0, wxyz = 0.0;
                    if (sy) {
                        wy = __ldcg(q + oy);
                        if (sx) wxy = __ldcg(q + ox + oy);
                    }
                    if (sz) {
                        wz = __ldcg(q + oz);
                        if (sx) wxz = __ldcg(q + ox + oz);
                        if (sy) {
                            wyz = __ldcg(q + oy + oz);
                            if (sx) wxyz = __ldcg(q + ox + oy + oz);
                        }
                    }
                    c[s] = wv[s] + wx;
                    if (sy) c[s] += wy + wxy;
                    if (sz) {
                        double cz = wz + wxz;
                        if (sy) cz += wyz + wxyz;
                        c[s] += cz;
                    }
                }
        }
        if (warp == 0) {
            pap = warp0_sum(s_red[0], min(ns, S::T));
            if (lane == 0) s_bc[0] = rho / pap;
        }
        __syncthreads();
        alpha = s_bc[0];
        // ---- r -= alpha (QQ^T w), <r, r> at each node's first copy
        double acc = 0.0, acc2 = 0.0;
        if (act) {
#pragma unroll
            for (int s = 0; s < KS; ++s)
                if (d + 3 * s < NQ) {
                    r[s] = fma(masked(s) ? 0.0 : -alpha, c[s], r[s]);
                    if (sx >= 0 && sy >= 0 && sz_of(s) >= 0) {
                        const double zr = PRE ? dv[PRE ? s : 0] * r[s] : r[s];
                        acc = fma(r[s], zr, acc);
                        if (PRE) acc2 = fma(r[s], r[s], acc2);
                    }
                }
        }
        s_red[0][tid] = acc;
        if (PRE) s_red[NV2 - 1][tid] = acc2;
        __syncthreads();
        double mine[NV2] = {};
        if (warp == 0) {
#pragma unroll
            for (int v = 0; v < NV2; ++v) mine[v] = warp0_sum(s_red[v], S::T);
        }
        // ---- second exchange: rho; x += alpha p meanwhile
        if (warp != 0) {
#pragma unroll
            for (int s = 0; s < KS; ++s) x[s] = fma(alpha, p[s], x[s]);
        }
        double share2[NV2];
        const bool ok2 = exchange<NV2, false>(slots2, nb, e, uint32_t(n), mine, share2, &ns, A.limit_ns);
        __syncthreads();       // warp 0 has read s_red
#pragma unroll
        for (int v = 0; v < NV2; ++v) s_red[v][tid] = share2[v];
        if (__syncthreads_or(!ok2)) {
            if (tid == 0) atomicExch(A.status, int32_t(kStatusExchangeTimeout));
            return;
        }
        if (warp == 0) {
            const double rho_new = warp0_sum(s_red[0], min(ns, S::T));
            rr = PRE ? warp0_sum(s_red[NV2 - 1], min(ns, S::T)) : rho_new;
            // both quotients in one division: beta in lane 0, rr / ref in lane 1
            const double rr0 = __shfl_sync(0xffffffffu, rr, 0);
            const double q = (lane == 0 ? rho_new : rr0) / (lane == 0 ? rho : ref);
            const bool conv = __shfl_sync(0xffffffffu, int(q <= t2), 1) != 0;
            ++iter;
            if (lane == 0) {
                if (hist && e == 0) hist[iter] = rr;   // its root at the end
                s_bc[1] = q;
                rho = rho_new;
                s_stop = conv || iter >= maxit;
            }
#pragma unroll
            for (int s = 0; s < KS; ++s) x[s] = fma(alpha, p[s], x[s]);
        }
        __syncthreads();
        beta = s_bc[1];
        if (s_stop || n == A.iters) break;
    }
    // p goes back to its buffer once every block has read the last w from it
    const double none[1] = {0.0};
    double share[1];
    int ns;
    if (__syncthreads_or(!exchange<1, true>(slots1, nb, e, uint32_t(n + 1), none, share, &ns, A.limit_ns))) {
        if (tid == 0) atomicExch(A.status, int32_t(kStatusExchangeTimeout));
        return;
    }
    if (act) {
#pragma unroll
        for (int s = 0; s < KS; ++s)
            if (d + 3 * s < NQ) {
                A.x[l0 + s * NT] = x[s];
                A.r[l0 + s * NT] = r[s];
                A.p[l0 + s * NT] = p[s];
            }
    }
    if (e == 0 && warp == 0 && hist) {
        __syncwarp();   // lane 0's stores
        for (int k = iter0 + 1 + lane; k <= iter; k += 32) hist[k] = sqrt(hist[k]);
    }
    if (e == 0 && tid == 0) {
        st->alpha = alpha;
        st->beta = beta;
        st->rho = rho;
        st->pap = pap;
        st->rr = rr;
        st->iter = iter;
        st->done = s_stop;
    }
}

// Iterations of one launch at most: the host checks the status in between.
constexpr int kSmallIters = 1024;

template <int NQ, bool PRE>
int small_capacity_nq(int *out) {
    using S = SmallShape<NQ>;
    static int blocks = 0;
    if (!blocks) {
        int per_sm = 0;
        const int rc = cuda_check(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, cg_small_kernel<NQ, PRE>, S::T,
                                                                                S::smem), "cg small: occupancy");
        if (rc != SEM_OK) return rc;
        blocks = per_sm * sm_count();
    }
    *out = blocks;
    return SEM_OK;
}

template <int NQ, bool PRE>
int launch_small_nq(const Problem *P, const SmallArgs &A, bool *refused) {
    using S = SmallShape<NQ>;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(unsigned(P->E));
    cfg.blockDim = dim3(unsigned(S::T));
    cfg.dynamicSmemBytes = S::smem;
    cfg.stream = stream();
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, cg_small_kernel<NQ, PRE>, A);
    if (err == cudaErrorCooperativeLaunchTooLarge) {
        cudaGetLastError();
        *refused = true;
        return SEM_OK;
    }
    count_launches(1);
    return cuda_check(err, "cg_small_kernel");
}

template <bool PRE>
int small_call(const Problem *P, const SmallArgs *A, bool *refused, int *capacity = nullptr) {
    switch (P->nq) {
#define SEM_SMALL(Q) \
    case Q: return A ? launch_small_nq<Q, PRE>(P, *A, refused) : small_capacity_nq<Q, PRE>(capacity);
        SEM_SMALL(2) SEM_SMALL(3) SEM_SMALL(4) SEM_SMALL(5) SEM_SMALL(6) SEM_SMALL(7) SEM_SMALL(8) SEM_SMALL(9) SEM_SMALL(10)
#undef SEM_SMALL
        default: return set_error(SEM_EARG, "cg: unsupported order");
    }
}

// Self-test of the exchange's bounded wait: gridDim.x blocks take part in an
// exchange of one more, whose slot nobody fills.
__global__ void exchange_probe_kernel(uint64_t *slots, int32_t *status, uint64_t limit_ns) {
    const double mine[1] = {1.0};
    double share[1];
    int n;
    const bool ok = exchange<1, true>(slots, int(gridDim.x) + 1, int(blockIdx.x), 1u, mine, share, &n, limit_ns);
    if (__syncthreads_or(!ok) && threadIdx.x == 0) atomicExch(status, int32_t(kStatusExchangeTimeout));
}

}  // namespace

// Problems this path takes: the fixed-point operator is the order's choice,
// every element has a resident block (152 SMs: 608 at N = 7, 456 at N = 8, 304
// at N = 9), and there are at most five per SM.  At the limit of residence this
// kernel is still the faster one (E = 600: N = 7 22.3 us an iteration against
// 23.1, N = 6 19.6 against 25.4, N = 4 14.9 against 19.6; E = 441, N = 8 22.2
// against 29.0); where small elements would allow more, the exchanges grow past
// it (E = 800, N = 3 15.7 against 16.1; E = 1728, N = 2 22 against 18; E = 4096,
// N = 1 53 against 16).
bool small_fits(const Problem *P, bool pre) {
    if (tune_get(kTuneF64, P->nq).variant != kAxLinesFX) return false;
    int capacity = 0;
    const int rc = pre ? small_call<true>(P, nullptr, nullptr, &capacity) : small_call<false>(P, nullptr, nullptr, &capacity);
    return rc == SEM_OK && P->E <= std::min<int64_t>(capacity, 5 * int64_t(sm_count()));
}

// One launch: up to kSmallIters iterations from P's state, x complete at its
// end (nothing deferred).  *refused: the launch's blocks cannot all be resident
// (fewer SMs than the device has, say), nothing ran.
int launch_small(const Problem *P, bool pre, bool *refused) {
    SmallArgs A{};
    A.x = P->x;
    A.r = P->r;
    A.p = P->p;
    A.w = P->w;
    A.dinv = P->dinv;
    A.G = P->Gfx;
    A.kg = P->kgfx;
    A.d = P->fxc->d;
    A.dt = P->fxc->dt;
    A.nx = P->nx;
    A.ny = P->ny;
    A.nz = P->nz;
    A.iters = kSmallIters;
    A.st = P->st;
    A.slots = reinterpret_cast<uint64_t *>(P->partials);
    A.status = status_word();
    A.limit_ns = kExchangeLimitNs;
    const int64_t words = 6 * (P->E + (P->E + 31) / 32);
    if (words > P->partials_cap) return set_error(SEM_ERANGE, "cg: more blocks than reduction slots");
    const int rc = cuda_check(cudaMemsetAsync(A.slots, 0, sizeof(uint64_t) * size_t(words), stream()), "cg: slots");
    if (rc != SEM_OK) return rc;
    *refused = false;
    return pre ? small_call<true>(P, &A, refused) : small_call<false>(P, &A, refused);
}

// Runs the exchange of 41 blocks with 40 of them (two groups, so that the
// leader's wait and the others' both run out, each after ~limit_ns).
int probe_exchange_timeout(uint64_t limit_ns) {
    if (limit_ns < 1000 || limit_ns > 100000000ull)
        return set_error(SEM_EARG, "exchange_probe: limit_ns must be in [1e3, 1e8]");
    constexpr unsigned kBlocks = 40;
    constexpr size_t kBytes = sizeof(uint64_t) * 2 * (kBlocks + 1 + 2);   // slots of the blocks and of two groups
    uint64_t *slots = static_cast<uint64_t *>(dev_alloc(kBytes));
    if (!slots) return SEM_ENOMEM;
    int rc = cuda_check(cudaMemsetAsync(slots, 0, kBytes, stream()), "exchange_probe: slots");
    if (rc == SEM_OK) {
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeCooperative;
        at.val.cooperative = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(kBlocks);
        cfg.blockDim = dim3(64);
        cfg.stream = stream();
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        count_launches(1);
        rc = cuda_check(cudaLaunchKernelEx(&cfg, exchange_probe_kernel, slots, status_word(), limit_ns),
                        "exchange_probe_kernel");
    }
    if (rc == SEM_OK) rc = cuda_check(cudaStreamSynchronize(stream()), "exchange_probe: sync");
    dev_free(slots);
    return rc;
}

}  // namespace sem
