// sem_ax_lines32.cu -- FP32 line operators for the inner solves of
// mixed-precision refinement, plain and CG, geometric factors in FP32 or BF16:
// the direct-load kernel (sem_ax_f32.cuh), and the line kernel with slab and
// factors staged in shared memory (sem_ax_lines.cuh).
#include <cuda_bf16.h>

#include <algorithm>

#include "sem_ax_f32.cuh"

namespace sem {

template <int NQ, typename GT, bool CG>
__global__ void __maxnreg__((F32Regs<NQ, GT>::value)) ax_f32_kernel(const __grid_constant__ AxLineArgs<float, GT> P) {
    extern __shared__ __align__(16) float smem32[];
    const AxArgs<float, GT> &A = P.a;
    const int64_t e0 = int64_t(blockIdx.x) * P.epb;
    const int ne = int(min(int64_t(P.epb), A.E - e0));
    pdl_wait();
    if (CG && A.st->done) return;   // solve finished: the rest of the graph is a no-op
    f32_prefetch<NQ>(A.G, e0, ne);
    const float part = lines_group_f32<NQ, GT, CG>(A.x, A.y, A.p, A.xs, A.G, P.d, P.dt, CG ? float(A.st->beta) : 0.f,
                                                   CG ? float(A.st->alpha) : 0.f, e0, ne, P.epb, smem32);
    if (CG) {
        // the threads' parts are added in FP64 at N <= 3, whose sums always were
        // (all orders: 0.3 to 0.7 us more an iteration)
        const double s = NQ <= 4 ? block_sum_wide(double(part), reinterpret_cast<double *>(smem32))
                                 : double(block_sum_f32(part, smem32));
        if (threadIdx.x == 0) A.partials[blockIdx.x] = s;
    }
}

__global__ void __launch_bounds__(kPapThreads) pap_sum_kernel(double *partials, int64_t cap, int n, CgState *st) {
    pdl_wait();
    if (st->done) return;
    pap_sum(partials, cap, n, int(blockIdx.x), int(gridDim.x), st);
}

// Elements per block: the tuned number, or fewer for problems that would not
// give every SM a block.
static int f32_epb(const Problem *P, int tuned) {
    return int(std::max<int64_t>(1, std::min<int64_t>(tuned, P->E / sm_count())));
}

template <int NQ, typename GT, bool CG>
static int launch_f32_nq(const Problem *Pb, const AxLineArgs<float, GT> &L) {
    const size_t sm = f32_smem<NQ>(L.epb);
    auto kern = ax_f32_kernel<NQ, GT, CG>;
    static size_t sm_set = 0;
    if (sm > sm_set) {   // not a stream operation: also fine during a capture
        const int rc = cuda_check(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm)),
                                  "ax f32: smem attribute");
        if (rc != SEM_OK) return rc;
        sm_set = sm;
    }
    const int64_t blocks = (Pb->E + L.epb - 1) / L.epb;
    if (CG && blocks > Pb->partials_cap) return set_error(SEM_ERANGE, "ax f32: more blocks than reduction slots");
    count_launches(1);
    int rc = cuda_check(launch_pdl(kern, unsigned(blocks), unsigned(line_threads(NQ, L.epb)), sm, L), "ax_f32_kernel");
    if (CG && rc == SEM_OK) {
        count_launches(1);
        rc = cuda_check(launch_pdl(pap_sum_kernel, unsigned(pap_blocks(blocks)), unsigned(kPapThreads), 0,
                                   L.a.partials, L.a.cap, int(blocks), L.a.st),
                        "pap_sum_kernel");
    }
    return rc;
}

template <typename GT, bool CG>
static int launch_f32_any(const Problem *Pb, const AxLineArgs<float, GT> &L) {
    switch (Pb->nq) {
        case 2: return launch_f32_nq<2, GT, CG>(Pb, L);
        case 3: return launch_f32_nq<3, GT, CG>(Pb, L);
        case 4: return launch_f32_nq<4, GT, CG>(Pb, L);
        case 5: return launch_f32_nq<5, GT, CG>(Pb, L);
        case 6: return launch_f32_nq<6, GT, CG>(Pb, L);
        case 7: return launch_f32_nq<7, GT, CG>(Pb, L);
        case 8: return launch_f32_nq<8, GT, CG>(Pb, L);
        case 9: return launch_f32_nq<9, GT, CG>(Pb, L);
        case 10: return launch_f32_nq<10, GT, CG>(Pb, L);
        default: return set_error(SEM_EARG, "ax f32: unsupported order");
    }
}

template <typename GT>
static int launch_lines32_gt(const Problem *P, const GT *G, const float *x, float *y, bool cg, int epb, bool staged) {
    if (!lines_epb_ok(P->nq, epb, sizeof(float), staged ? 6 * int(sizeof(GT)) : 0))
        return set_error(SEM_EARG, "ax lines: bad elements per block");
    AxArgs<float, GT> a = ax_args<float, GT>(P, G, P->partials, P->st_in);
    a.x = cg ? P->r32 : x;
    a.y = cg ? P->w32 : y;
    if (cg) {
        a.p = P->p32;
        a.xs = f32_defers(P->nq, sizeof(GT) == 4 ? kGF32 : kGBF16) ? P->d32 : nullptr;   // d += alpha p of the previous iteration
    }
    const AxLineArgs<float, GT> L = line_args(a, P->oc.D, P->nq, staged ? epb : f32_epb(P, epb));
    if (staged)
        return cg ? launch_lines_any<float, GT, true, false, kGStaged>(P, L)
                  : launch_lines_any<float, GT, false, false, kGStaged>(P, L);
    return cg ? launch_f32_any<GT, true>(P, L) : launch_f32_any<GT, false>(P, L);
}

int launch_lines32(const Problem *P, const float *x, float *y, int gprec, bool cg, int epb, bool staged) {
    if (gprec == kGF32) return launch_lines32_gt(P, static_cast<const float *>(P->G32), x, y, cg, epb, staged);
    return launch_lines32_gt(P, static_cast<const __nv_bfloat16 *>(P->G16), x, y, cg, epb, staged);
}

}  // namespace sem
