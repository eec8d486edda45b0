// sem_ax_dw.cu -- the double-word CG operator (sem_ax_dw.cuh): its geometric
// factors in double-word form, its coefficients and its launches, for every
// order.
#include "sem_ax_dw.cuh"

namespace sem {

// Gdw[2 (6 l + c)] = rn(G), Gdw[2 (6 l + c) + 1] = rn(G - rn(G)); *top the
// largest |G|'s upper half.
__global__ void geometry_dw_kernel(const double *__restrict__ G, float *__restrict__ Gdw, int64_t n, uint32_t *top) {
    uint32_t mx = 0;
    for (int64_t q = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; q < n; q += int64_t(gridDim.x) * blockDim.x) {
        const double g = G[q];
        const float h = __double2float_rn(g);
        Gdw[2 * q] = h;
        Gdw[2 * q + 1] = __double2float_rn(g - double(h));
        mx = max(mx, uint32_t(__double2hiint(g)) & 0x7fffffffu);
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0) atomicMax(top, mx);
}

// The factors in double-word form (made once), unless the problem's are outside
// FP32's exponents with room for the low parts (Gdw then stays null).  Uses the
// partials buffer; synchronises the first time.
int dw_prepare(Problem *P) {
    if (P->Gdw || P->dw_out) return SEM_OK;
    const size_t bytes = sizeof(float) * 12 * size_t(P->nL);
    float *g = static_cast<float *>(dev_alloc(bytes));
    if (!g && P->Gfx) {   // both forms do not fit: the other one is made again when it is needed
        cudaStreamSynchronize(stream());
        problem_drop_graph(&P->graph);
        problem_drop_graph(&P->graph_pcg);
        fx_release(P);
        g = static_cast<float *>(dev_alloc(bytes));
    }
    if (!g) return SEM_ENOMEM;
    const int64_t n = 6 * P->nL;
    const unsigned blocks = unsigned(std::min<int64_t>((n + 255) / 256, int64_t(sm_count()) * 16));
    uint32_t *top = reinterpret_cast<uint32_t *>(P->partials);
    int rc = cuda_check(cudaMemsetAsync(top, 0, sizeof(uint32_t), stream()), "geometry_dw: largest factor");
    if (rc == SEM_OK) {
        geometry_dw_kernel<<<blocks, 256, 0, stream()>>>(P->G, g, n, top);
        count_launches(1);
        rc = cuda_check(cudaGetLastError(), "geometry_dw_kernel");
    }
    if (rc == SEM_OK)
        rc = cuda_check(cudaMemcpyAsync(&P->st_host->pad0, top, sizeof(uint32_t), cudaMemcpyDeviceToHost, stream()),
                        "geometry_dw: largest factor");
    if (rc == SEM_OK) rc = cuda_check(cudaStreamSynchronize(stream()), "geometry_dw: sync");
    const int e = int(uint32_t(P->st_host->pad0) >> 20) - 1023;
    P->dw_out = rc == SEM_OK && (e < -60 || e > 60);
    if (rc != SEM_OK || P->dw_out) {
        dev_free(g);
        return rc;
    }
    P->Gdw = g;
    return SEM_OK;
}

void dw_release(Problem *P) {
    if (P->Gdw) dev_free(P->Gdw);
    P->Gdw = nullptr;
}

// Elements per block: part of the summation order of <p, A p>, hence fixed per
// order (the fastest of the former tuner's candidates at 1.7e7 nodes).
static int dw_epb(int nq) {
    constexpr int epb[kMaxQ + 1] = {0, 0, 32, 14, 8, 5, 7, 5, 4, 3, 5};
    return epb[nq];
}

template <int NQ>
static int launch_dw_nq(const Problem *Pb, const AxDwArgs &L) {
    const int nt = line_threads(NQ, L.epb);
    const size_t sm = LineShape::smem(NQ, L.epb, int(sizeof(double)));
    auto kern = ax_dw_kernel<NQ>;
    // the dynamic shared-memory limit, raised by the first launch of an order
    static bool sm_set = false;
    if (!sm_set) {
        const int rc = cuda_check(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm)),
                                  "ax dw: smem attribute");
        if (rc != SEM_OK) return rc;
        sm_set = true;
    }
    const int64_t blocks = (Pb->E + L.epb - 1) / L.epb;
    if (blocks > Pb->partials_cap) return set_error(SEM_ERANGE, "ax dw: more blocks than reduction slots");
    kern<<<unsigned(blocks), nt, sm, stream()>>>(L);
    count_launches(1);
    return cuda_check(cudaGetLastError(), "ax_dw_kernel");
}

int launch_ax_dw(const Problem *P) {
    if (!P->Gdw) return set_error(SEM_EARG, "ax dw: double-word factors not prepared (dw_prepare)");
    AxDwArgs L{};
    L.r = P->r;
    L.w = P->w;
    L.p = P->p;
    L.xs = P->x;   // x += alpha p of the previous iteration
    L.Gdw = P->Gdw;
    L.partials = P->partials;
    L.st = P->st;
    L.status = status_word();
    L.E = P->E;
    L.cap = P->partials_cap;
    double Dt[kMaxQ * kMaxQ];
    for (int i = 0; i < P->nq; ++i)
        for (int l = 0; l < P->nq; ++l) Dt[i * P->nq + l] = P->oc.D[l * P->nq + i];
    L.d = eo_coefficients_dw(P->oc.D, P->nq);
    L.dt = eo_coefficients_dw(Dt, P->nq);
    L.epb = dw_epb(P->nq);
    switch (P->nq) {
        case 2: return launch_dw_nq<2>(P, L);
        case 3: return launch_dw_nq<3>(P, L);
        case 4: return launch_dw_nq<4>(P, L);
        case 5: return launch_dw_nq<5>(P, L);
        case 6: return launch_dw_nq<6>(P, L);
        case 7: return launch_dw_nq<7>(P, L);
        case 8: return launch_dw_nq<8>(P, L);
        case 9: return launch_dw_nq<9>(P, L);
        case 10: return launch_dw_nq<10>(P, L);
        default: return set_error(SEM_EARG, "ax dw: unsupported order");
    }
}

}  // namespace sem
