// sem_ax_fx.cu -- the fixed-point FP64 operator (sem_ax_fx.cuh): its geometric
// factors as integers, its coefficients, and its launches (plain y =
// A_local x, the CG operator and the Jacobi-PCG operator, for every order).
#include <algorithm>

#include "sem_ax_fx.cuh"
#include "sem_device.cuh"

namespace sem {

// One block per element: the largest exponent of the element's factors, then
// g 2^kg rounded to integers, |G| < 2^kFxGBits, in integer arithmetic (FP64
// conversions run at 1/64 rate), with fewer bits where the element's sum of
// <x, y> could pass 63 (FxBound; elements with vertices moved by up to 0.6 of a
// side reach 0.39 of the limit, at N = 9).  Bound by HBM: 48 B read and written
// per node; the later reads hit L1 or L2.
__global__ void __launch_bounds__(256) geometry_fx_kernel(const double *__restrict__ G, int4 *__restrict__ out,
                                                          int32_t *__restrict__ kg, int nq, int64_t E, FxBound B) {
    __shared__ uint32_t s_max;
    __shared__ float s_sum[32];
    __shared__ int s_less;
    const int np = nq * nq * nq;
    for (int64_t e = blockIdx.x; e < E; e += gridDim.x) {
        __syncthreads();
        if (threadIdx.x == 0) s_max = uint32_t(kFxEmin) << 20;
        __syncthreads();
        const double2 *g = reinterpret_cast<const double2 *>(G + 6 * e * np);
        uint32_t mx = 0;
        for (int q = threadIdx.x; q < 3 * np; q += blockDim.x) {
            const double2 t = __ldg(g + q);
            mx = max(mx, max(uint32_t(__double2hiint(t.x)) & 0x7fffffffu, uint32_t(__double2hiint(t.y)) & 0x7fffffffu));
        }
        mx = __reduce_max_sync(0xffffffffu, mx);
        if ((threadIdx.x & 31) == 0) atomicMax(&s_max, mx);
        __syncthreads();
        int emax = int(s_max >> 20);
        // |g| of the largest exponent in [1, 2), to 20 bits
        auto rel = [emax](double d) {
            const int h = __double2hiint(d) & 0x7fffffff;
            return (h >> 20) - emax + 127 > 0 ? __int_as_float((h - ((emax - 127) << 20)) << 3) : 0.f;
        };
        float sum = 0.f;
        for (int node = threadIdx.x; node < np; node += blockDim.x) {
            const double2 a = __ldg(g + 3 * node), b = __ldg(g + 3 * node + 1), c = __ldg(g + 3 * node + 2);
            const float r = B.rows[node % nq], s = B.rows[node / nq % nq], t = B.rows[node / nq / nq];
            sum += r * r * rel(a.x) + s * s * rel(b.y) + t * t * rel(c.y) +
                   2.f * (r * s * rel(a.y) + r * t * rel(b.x) + s * t * rel(c.x));
        }
        sum = block_sum_f32(sum, s_sum);
        if (threadIdx.x == 0) {
            int less = 0;
            while (sum > B.limit && less < 8) {
                sum *= 0.5f;
                ++less;
            }
            s_less = less;
        }
        __syncthreads();
        emax += s_less;
        if (threadIdx.x == 0) kg[e] = kFxGBits - 53 + 1075 - emax;
        auto fix = [emax](double d) {
            const int64_t bits = __double_as_longlong(d);
            const int hi = int(bits >> 32);
            const int s = min(emax - int((uint32_t(hi) << 1) >> 21), 63);
            const uint64_t m = (uint64_t(uint32_t((hi & 0xfffff) | 0x100000)) << 32) | uint32_t(bits);
            const int64_t v = int64_t(((m << (kFxGBits - 53)) + (s ? uint64_t(1) << (s - 1) : 0)) >> s);
            return fx_limbs(hi < 0 ? -v : v);
        };
        int4 *o = out + e * (3 * np);
        for (int q = threadIdx.x; q < 3 * np; q += blockDim.x) {
            const double2 t = __ldg(g + q);
            const fxl a = fix(t.x), b = fix(t.y);
            const int node = q / 3;
            o[(q - 3 * node) * np + node] = make_int4(a.h, a.l, b.h, b.l);
        }
    }
}

int fx_prepare(Problem *P) {
    if (P->Gfx) return SEM_OK;
    int4 *g = static_cast<int4 *>(dev_alloc(sizeof(int4) * 3 * size_t(P->nL)));
    if (!g && P->Gdw) {   // both forms do not fit: the other one is made again when it is needed
        cudaStreamSynchronize(stream());
        problem_drop_graph(&P->graph_steps);
        dw_release(P);
        g = static_cast<int4 *>(dev_alloc(sizeof(int4) * 3 * size_t(P->nL)));
    }
    int32_t *kg = static_cast<int32_t *>(dev_alloc(sizeof(int32_t) * size_t(P->E)));
    int rc = g && kg ? SEM_OK : SEM_ENOMEM;
    if (rc == SEM_OK) {
        const unsigned blocks = unsigned(std::min<int64_t>(P->E, int64_t(sm_count()) * 32));
        FxConsts c;
        fx_coefficients(P->oc.D, P->nq, &c.d, &c.dt);
        geometry_fx_kernel<<<blocks, 256, 0, stream()>>>(P->G, g, kg, P->nq, P->E,
                                                         fx_bound(P->oc.D, P->nq, c.d.k, c.dt.k));
        count_launches(1);
        rc = cuda_check(cudaGetLastError(), "geometry_fx_kernel");
    }
    if (rc != SEM_OK) {
        if (g) dev_free(g);
        if (kg) dev_free(kg);
        return rc;
    }
    P->Gfx = g;
    P->kgfx = kg;
    P->fxc = new FxConsts();
    fx_coefficients(P->oc.D, P->nq, &P->fxc->d, &P->fxc->dt);
    return SEM_OK;
}

void fx_release(Problem *P) {
    if (P->Gfx) dev_free(P->Gfx);
    if (P->kgfx) dev_free(P->kgfx);
    delete P->fxc;
    P->Gfx = nullptr;
    P->kgfx = nullptr;
    P->fxc = nullptr;
}

// Elements per block: the tuned number, or fewer for problems that would not
// give every SM a block (E = 64, N = 7: 64 blocks of one element instead of
// 16 of four).
static int fx_epb(const Problem *P, int tuned) {
    return int(std::max<int64_t>(1, std::min<int64_t>(tuned, P->E / sm_count())));
}

template <int NQ, bool CG, bool PRE>
static int launch_fx_nq(const Problem *Pb, const AxFxArgs &L) {
    const int nt = line_threads(NQ, L.epb);
    const size_t sm = fx_smem<NQ>(L.epb);
    auto kern = ax_fx_kernel<NQ, CG, PRE>;
    // raise the dynamic shared-memory limit when a larger block is first
    // asked for (the tuner and the first solve do so before any capture)
    static size_t sm_set = 0;
    if (sm > sm_set) {
        const int rc = cuda_check(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm)),
                                  "ax fx: smem attribute");
        if (rc != SEM_OK) return rc;
        sm_set = sm;
    }
    const int64_t blocks = (Pb->E + L.epb - 1) / L.epb;
    if (CG && blocks > Pb->partials_cap) return set_error(SEM_ERANGE, "ax fx: more blocks than reduction slots");
    count_launches(1);
    return cuda_check(launch_pdl(kern, unsigned(blocks), unsigned(nt), sm, L), "ax_fx_kernel");
}

template <bool CG, bool PRE>
static int launch_fx_any(const Problem *Pb, const AxFxArgs &L) {
    switch (Pb->nq) {
        case 2: return launch_fx_nq<2, CG, PRE>(Pb, L);
        case 3: return launch_fx_nq<3, CG, PRE>(Pb, L);
        case 4: return launch_fx_nq<4, CG, PRE>(Pb, L);
        case 5: return launch_fx_nq<5, CG, PRE>(Pb, L);
        case 6: return launch_fx_nq<6, CG, PRE>(Pb, L);
        case 7: return launch_fx_nq<7, CG, PRE>(Pb, L);
        case 8: return launch_fx_nq<8, CG, PRE>(Pb, L);
        case 9: return launch_fx_nq<9, CG, PRE>(Pb, L);
        case 10: return launch_fx_nq<10, CG, PRE>(Pb, L);
        default: return set_error(SEM_EARG, "ax fx: unsupported order");
    }
}

int launch_lines_fx(const Problem *P, const double *x, double *y, int mode, int epb) {
    if (!lines_epb_ok(P->nq, epb, sizeof(double))) return set_error(SEM_EARG, "ax fx: bad elements per block");
    if (!P->Gfx) return set_error(SEM_EARG, "ax fx: integer factors not prepared (fx_prepare)");
    AxFxArgs L{};
    L.a = ax_args<double, double>(P, P->G, P->partials, P->st);
    L.G = P->Gfx;
    L.kg = P->kgfx;
    L.d = P->fxc->d;
    L.dt = P->fxc->dt;
    L.epb = fx_epb(P, epb);
    if (mode == 0) {
        L.a.x = x;
        L.a.y = y;
        return launch_fx_any<false, false>(P, L);
    }
    L.a.x = P->r;
    L.a.y = P->w;
    L.a.p = P->p;
    L.a.xs = P->x;   // x += alpha p of the previous iteration
    if (mode == 1) return launch_fx_any<true, false>(P, L);
    L.a.dinv = P->dinv;
    return launch_fx_any<true, true>(P, L);
}

}  // namespace sem
