// sem_ax.cu -- FP64 local Poisson operator: the column kernel's
// instantiations (sem_ax_kernel.cuh) -- plain y = A_local x, the CG variant
// with the fused p-update and <p, A p> reduction, the Jacobi-PCG variant --
// and the dispatch to the variant the per-order tuner chose (the line kernel
// lives in sem_ax_lines64.cu, its fixed-point form in sem_ax_fx.cu).
#include "sem_ax_kernel.cuh"

namespace sem {

int prepare_ax(const Problem *Pb) { return prepare_ax_any<double, double>(Pb); }

int prepare_f64_variant(Problem *P) {
    return tune_get(kTuneF64, P->nq).variant == kAxLinesFX ? fx_prepare(P) : SEM_OK;
}

// The fixed-point variant's factors: made on first use outside a capture
// (solves prepare them before capturing their graphs).
static int ensure_fx(const Problem *Pb) {
    if (Pb->Gfx) return SEM_OK;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    const int rc = cuda_check(cudaStreamIsCapturing(stream(), &cs), "ax fx: capture status");
    if (rc != SEM_OK) return rc;
    if (cs != cudaStreamCaptureStatusNone)
        return set_error(SEM_EARG, "ax fx: integer factors must be prepared before a capture");
    return fx_prepare(const_cast<Problem *>(Pb));
}

int launch_ax(const Problem *Pb, const double *x, double *y) {
    const TuneChoice c = tune_get(kTuneF64, Pb->nq);
    if (c.variant == kAxLinesFX) {
        const int rc = ensure_fx(Pb);
        return rc != SEM_OK ? rc : launch_lines_fx(Pb, x, y, 0, c.epb);
    }
    if (c.variant == kAxLines) return launch_lines64(Pb, x, y, 0, c.epb);
    AxArgs<double, double> a = ax_args<double, double>(Pb, Pb->G, Pb->partials, Pb->st);
    a.x = x;
    a.y = y;
    return launch_ax_any<double, double, false>(Pb, a);
}

int launch_ax_cg(const Problem *Pb) {
    const TuneChoice c = tune_get(kTuneF64, Pb->nq);
    if (c.variant == kAxLinesFX) {
        const int rc = ensure_fx(Pb);
        return rc != SEM_OK ? rc : launch_lines_fx(Pb, nullptr, nullptr, 1, c.epb);
    }
    if (c.variant == kAxLines) return launch_lines64(Pb, nullptr, nullptr, 1, c.epb);
    AxArgs<double, double> a = ax_args<double, double>(Pb, Pb->G, Pb->partials, Pb->st);
    a.x = Pb->r;
    a.y = Pb->w;
    a.p = Pb->p;
    a.xs = Pb->x;   // x += alpha p of the previous iteration
    return launch_ax_any<double, double, true>(Pb, a);
}

int launch_ax_pcg(const Problem *Pb) {
    const TuneChoice c = tune_get(kTuneF64, Pb->nq);
    if (c.variant == kAxLinesFX) {
        const int rc = ensure_fx(Pb);
        return rc != SEM_OK ? rc : launch_lines_fx(Pb, nullptr, nullptr, 2, c.epb);
    }
    if (c.variant == kAxLines) return launch_lines64(Pb, nullptr, nullptr, 2, c.epb);
    AxArgs<double, double> a = ax_args<double, double>(Pb, Pb->G, Pb->partials, Pb->st);
    a.x = Pb->r;
    a.y = Pb->w;
    a.p = Pb->p;
    a.xs = Pb->x;   // x += alpha p of the previous iteration
    a.dinv = Pb->dinv;
    return launch_ax_any<double, double, true, true>(Pb, a);
}

}  // namespace sem
