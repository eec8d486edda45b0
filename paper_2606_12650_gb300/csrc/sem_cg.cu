// sem_cg.cu -- direct-stiffness sum, Dirichlet mask, weighted dot product and
// the device-resident conjugate-gradient driver.
//
// Gather-scatter (the paper's "gs" kernel, Section V-B: an outer loop over
// global ids split across blocks and threads, and order-enforced inner loops
// over the copies).  Each thread owns one global node that has two or more
// copies; it adds the copies in ascending local index and writes the sum back
// to each.  There are no floating-point atomics, so the result does not
// depend on scheduling and matches an ascending sequential sum bit for bit.
//
// CG (Nekbone without preconditioner, Section VIII-A).  One iteration is two
// kernels:
//   1. the operator kernel in CG mode (the variant the tuner chose): the
//      previous iteration's x += alpha p, then p = r + beta p; w = A_local p;
//      <p, A p>; alpha
//   2. cg_update_owner_kernel (sem_box.cuh): the first copy of every global
//      node sums the copies of w (the direct-stiffness sum, in a fixed order),
//      applies r -= alpha (QQ^T w) and writes the result to every copy; <r, r>
//      is accumulated once per global node; the block that completes the grid
//      sum forms rho, beta, the iteration count and the stop flag.
// Moving x += alpha p into the next operator kernel (which has p in shared
// memory anyway) takes 24 of the update's 48 bytes per node off HBM and one
// FP64 operation off the update; x_finish_kernel applies the last one.
// The dot products of the paper are tree reductions (Section VIII-B, the
// unrolled reduction of Table "HIP-variable vs HIP-fixed"); here each block
// reduces in a fixed order, the last block of each group of blocks sums the
// group's partials in index order and the last group sums the group sums
// (grid_sum), so results are reproducible run to run.  Scalars
// never leave the device inside the loop: the host replays a CUDA graph of K
// iterations and polls the stop flag once per replay.  Problems of up to five
// elements per SM run in one kernel instead (sem_cg_small.cu), and solves of a
// given number of iterations (tol = 0) keep their own operator, update and
// summation orders (sem_ax_dw.cuh says why).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>

#include "sem_box.cuh"
#include "sem_device.cuh"
#include "sem_internal.h"

namespace sem {

constexpr int kThreads = 256;

static unsigned grid_for(int64_t n, int threads) {
    int64_t b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    return unsigned(b);
}

// ---------------------------------------------------------------- gs / mask
// u = QQ^T u, or mask(QQ^T u), in place.  A global node's first copy (no
// neighbour across a low face) adds its copies -- per direction its own
// element and, across a high face, the next one -- in ascending local index
// and writes the sum to each: every value is read and written by that one
// thread.  The copies follow from the box structure, so no index lists are
// read.  One thread per node on an element's high faces, in the order all
// faces (1 addition), all edges (3), all corners (7): a warp runs the
// additions of one class (predicated off they would cost as much on the
// 1/64-rate FP64 pipe: 200 us at E = 32^3, N = 7 with one thread per node and
// all seven, 66 us from index lists plus 4 us for the mask's).  MASK: nodes of
// the cube's high faces are zeroed by their own thread, those of its low faces
// by the last NQ^2 (ny nz + nx nz + nx ny) threads.
template <int M>
__device__ __forceinline__ void sum_copies(double *u, const int (&o)[M]) {
    constexpr int C = 1 << M;
    double v[C];
    int at[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
        at[c] = 0;
#pragma unroll
        for (int d = 0; d < M; ++d)
            if (c >> d & 1) at[c] += o[d];
        v[c] = __ldcg(u + at[c]);
    }
    double s = v[0];
#pragma unroll
    for (int c = 1; c < C; ++c) s += v[c];
#pragma unroll
    for (int c = 0; c < C; ++c) u[at[c]] = s;
}

template <int NQ, bool MASK>
__global__ void __launch_bounds__(256) gs_box_kernel(double *u, int64_t E, BoxDims bd, int64_t total) {
    constexpr int N = NQ - 1, N2 = N * N, NQ2 = NQ * NQ, NP = NQ2 * NQ;
    const int64_t t64 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    pdl_wait();
    if (t64 >= total) return;
    const unsigned nE = unsigned(E);
    unsigned t = unsigned(t64), e;
    int c[3], m;                       // (i, j, k), the number of them at N by class
    if (t < nE * (3 * N2)) {           // faces
        e = t / (3 * N2);
        const int f = int(t - e * (3 * N2)), d = f / N2, r = f - d * N2, q = r / N, p = r - q * N;
        c[0] = d == 0 ? N : p;
        c[1] = d == 1 ? N : (d == 0 ? p : q);
        c[2] = d == 2 ? N : q;
        m = 1;
    } else if ((t -= nE * (3 * N2)) < nE * (3 * N)) {   // edges
        e = t / (3 * N);
        const int f = int(t - e * (3 * N)), d = f / N, p = f - d * N;
        c[0] = d == 0 ? p : N;
        c[1] = d == 1 ? p : N;
        c[2] = d == 2 ? p : N;
        m = 2;
    } else if ((t -= nE * (3 * N)) < nE) {              // corners
        e = t;
        c[0] = c[1] = c[2] = N;
        m = 3;
    } else {                                            // MASK: the cube's low faces
        t -= nE;
        const unsigned yz = unsigned(bd.ny * bd.nz) * NQ2, xz = unsigned(bd.nx * bd.nz) * NQ2;
        const int d = t < yz ? 0 : (t < yz + xz ? 1 : 2);
        if (d) t -= d == 1 ? yz : yz + xz;
        const unsigned g = t / NQ2;
        const int r = int(t - g * NQ2), q = r / NQ, p = r - q * NQ;
        const unsigned n0 = unsigned(d == 0 ? bd.ny : bd.nx);
        const unsigned h = g / n0, a = g - h * n0;
        e = d == 0 ? a * unsigned(bd.nx) + h * unsigned(bd.nx * bd.ny)
                   : (d == 1 ? a + h * unsigned(bd.nx * bd.ny) : a + h * unsigned(bd.nx));
        const int i = d == 0 ? 0 : p, j = d == 1 ? 0 : (d == 0 ? p : q), k = d == 2 ? 0 : q;
        u[int64_t(e) * NP + k * NQ2 + j * NQ + i] = 0.0;
        return;
    }
    const unsigned g = divu(e, bd.dx);
    const int ex = int(e - g * unsigned(bd.nx));
    const unsigned tz = divu(g, bd.dy);
    const int ey = int(g - tz * unsigned(bd.ny)), ez = int(tz);
    const int pos[3] = {ex, ey, ez}, top[3] = {bd.nx - 1, bd.ny - 1, bd.nz - 1};
    const int off[3] = {NP - N, bd.nx * NP - N * NQ, bd.nx * bd.ny * NP - N * NQ2};
    double *v = u + int64_t(e) * NP + c[2] * NQ2 + c[1] * NQ + c[0];
    int o[3], n = 0;                   // offsets across the high faces with a neighbour, r first
    bool low = false, edge = false;    // a copy below; on a low face of the cube
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        if (c[d] == 0) (pos[d] > 0 ? low : edge) = true;
        if (c[d] == N && pos[d] < top[d]) {
            o[2] = n == 2 ? off[d] : 0;
            if (n == 1) o[1] = off[d];
            if (n == 0) o[0] = off[d];
            ++n;
        }
    }
    if (MASK) {
        if (n < m) {                   // on a high face of the cube
            *v = 0.0;
            return;
        }
        if (edge) return;
    }
    if (low || n == 0) return;
    if (n == 1) sum_copies<1>(v, {o[0]});
    else if (n == 2) sum_copies<2>(v, {o[0], o[1]});
    else sum_copies<3>(v, {o[0], o[1], o[2]});
}

template <int NQ>
static int launch_gs_nq(const Problem *P, double *u, bool mask) {
    const BoxDims bd = box_dims(P->nx, P->ny, P->nz);
    constexpr int N = NQ - 1;
    const int64_t nx = P->nx, ny = P->ny, nz = P->nz;
    int64_t total = P->E * (3 * N * N + 3 * N + 1);
    if (mask) total += NQ * NQ * (ny * nz + nx * nz + nx * ny);
    count_launches(1);
    return cuda_check(launch_pdl(mask ? gs_box_kernel<NQ, true> : gs_box_kernel<NQ, false>, grid_for(total, kThreads),
                                 kThreads, 0, u, P->E, bd, total),
                      "gs_box_kernel");
}

static int launch_gs_any(const Problem *P, double *u, bool mask) {
    switch (P->nq) {
        case 2: return launch_gs_nq<2>(P, u, mask);
        case 3: return launch_gs_nq<3>(P, u, mask);
        case 4: return launch_gs_nq<4>(P, u, mask);
        case 5: return launch_gs_nq<5>(P, u, mask);
        case 6: return launch_gs_nq<6>(P, u, mask);
        case 7: return launch_gs_nq<7>(P, u, mask);
        case 8: return launch_gs_nq<8>(P, u, mask);
        case 9: return launch_gs_nq<9>(P, u, mask);
        case 10: return launch_gs_nq<10>(P, u, mask);
        default: return set_error(SEM_EARG, "gs: unsupported order");
    }
}

__global__ void mask_kernel(double *__restrict__ u, const int32_t *__restrict__ idx, int64_t n) {
    const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (t < n) u[idx[t]] = 0.0;
}

// u = QQ^T u from the index lists: one thread per shared global id, its copies
// in ascending local index.
__global__ void gs_lists_kernel(double *__restrict__ u, const int32_t *__restrict__ ptr,
                                const int32_t *__restrict__ idx, int64_t nseg) {
    const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (t >= nseg) return;
    const int32_t b0 = ptr[t], b1 = ptr[t + 1];
    double s = u[idx[b0]];
    for (int32_t q = b0 + 1; q < b1; ++q) s += u[idx[q]];
    for (int32_t q = b0; q < b1; ++q) u[idx[q]] = s;
}

// N = 1 and 2 without the mask from the lists (where they exist) unless small:
// most of their nodes are corners and edges, whose copies the box form enumerates
// with more address arithmetic than the lists take to read (lists / box form, us:
// N = 1 1.7e7 nodes 115 / 145, 6e5 8.3 / 9.4, 2e5 6.2 / 5.7, 2e4 6.1 / 4.2; N = 2
// 6e5 10.6 / 13.2, 2e5 6.5 / 8.0, 2e4 6.1 / 4.7; from N = 3 on the box form is
// equal or faster, e.g. N = 7 66 / 52).
int launch_gs(const Problem *P, double *u) {
    const bool lists = P->maps_ready && ((P->nq == 2 && P->nL >= 300000) || (P->nq == 3 && P->nL >= 100000));
    if (!lists) return launch_gs_any(P, u, false);
    if (P->n_sh == 0) return SEM_OK;
    gs_lists_kernel<<<grid_for(P->n_sh, kThreads), kThreads, 0, stream()>>>(u, P->sh_ptr, P->sh_idx, P->n_sh);
    count_launches(1);
    return cuda_check(cudaGetLastError(), "gs_lists_kernel");
}

int launch_mask(const Problem *P, double *u) {
    if (P->n_mask == 0) return SEM_OK;
    mask_kernel<<<grid_for(P->n_mask, kThreads), kThreads, 0, stream()>>>(u, P->msk_idx, P->n_mask);
    count_launches(1);
    return cuda_check(cudaGetLastError(), "mask_kernel");
}

// mask(QQ^T u).  One pass of the box form, but at N = 1 from 6e6 nodes on the two
// lists (right-hand side of 1.7e7 nodes 218 -> 193 us, assembled operator 346 ->
// 320; 6e6 78.5 -> 76.6, 2e6 26 -> 29).
int launch_gs_mask(const Problem *P, double *u) {
    if (P->nq != 2 || !P->maps_ready || P->nL < 6000000) return launch_gs_any(P, u, true);
    const int rc = launch_gs(P, u);
    return rc != SEM_OK ? rc : launch_mask(P, u);
}

// ---------------------------------------------------------------- weighted dot
__global__ void dot_kernel(const double *__restrict__ c, const double *__restrict__ u,
                           const double *__restrict__ v, int64_t n, double *partials,
                           CgState *st) {
    __shared__ double red[32];
    double acc = 0.0;
    for (int64_t l = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; l < n;
         l += int64_t(gridDim.x) * blockDim.x)
        acc = fma(c[l] * u[l], v[l], acc);
    const double bs = block_sum(acc, red);
    if (publish_partial(bs, partials, &st->ticket_dot)) {
        const double tot = finish_partials(partials, int(gridDim.x), &st->ticket_dot, red);
        if (threadIdx.x == 0) st->dot_out = tot;
    }
}

static unsigned stream_grid(int64_t n) {
    // enough blocks to fill 152 SMs several times over, capped by the partials buffer
    int64_t b = (n + kThreads - 1) / kThreads;
    if (b > 152 * 8) b = 152 * 8;
    if (b < 1) b = 1;
    return unsigned(b);
}

int launch_dot(const Problem *P, const double *u, const double *v) {
    dot_kernel<<<stream_grid(P->nL), kThreads, 0, stream()>>>(P->c, u, v, P->nL, P->partials, P->st);
    count_launches(1);
    return cuda_check(cudaGetLastError(), "dot_kernel");
}

__global__ void sub_kernel(const double *__restrict__ a, const double *__restrict__ b,
                           double *__restrict__ out, int64_t n) {
    const int64_t l = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (l < n) out[l] = a[l] - b[l];
}

int launch_sub(const Problem *P, const double *a, const double *b, double *out) {
    sub_kernel<<<grid_for(P->nL, kThreads), kThreads, 0, stream()>>>(a, b, out, P->nL);
    count_launches(1);
    return cuda_check(cudaGetLastError(), "sub_kernel");
}

// ---------------------------------------------------------------- CG
// x = 0, p = 0, r = b; rho0 = <b, b>_c (weighted, local); scalars reset.
// steps: for the kernels of a given number of iterations.
__global__ void cg_init_kernel(const double *__restrict__ b, const double *__restrict__ c,
                               double *__restrict__ x, double *__restrict__ r,
                               double *__restrict__ p, int64_t n, double *partials, CgState *st,
                               int maxit, double tol, double *hist, bool steps) {
    __shared__ double red[32];
    double acc = 0.0;
    reset_group_tickets(partials);
    for (int64_t l = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; l < n;
         l += int64_t(gridDim.x) * blockDim.x) {
        const double bl = b[l];
        x[l] = 0.0;
        p[l] = 0.0;
        r[l] = bl;
        acc = fma(c[l] * bl, bl, acc);
    }
    const double bs = block_sum(acc, red);
    if (publish_partial(bs, partials, &st->ticket_dot)) {
        const double rho0 = finish_partials(partials, int(gridDim.x), &st->ticket_dot, red);
        if (threadIdx.x == 0) {
            st->rho = rho0;
            st->rho0 = rho0;
            st->alpha = 0.0;
            st->beta = 0.0;
            st->pap = 0.0;
            st->tol = tol;
            st->hist = hist;
            st->iter = 0;
            st->maxit = maxit;
            st->done = (rho0 == 0.0 || maxit <= 0) ? 1 : (steps && !dw_in_range(rho0) ? int(kDoneOutOfRange) : 0);
            st->ticket_ax = 0;
            st->ticket_up = 0;
            if (hist) hist[0] = sqrt(rho0);
        }
    }
}

int launch_cg_init(const Problem *P, const double *b, int maxit, double tol, double *hist, bool steps) {
    cg_init_kernel<<<stream_grid(P->nL), kThreads, 0, stream()>>>(b, P->c, P->x, P->r, P->p, P->nL,
                                                                   P->partials, P->st, maxit, tol, hist, steps);
    count_launches(1);
    return cuda_check(cudaGetLastError(), "cg_init_kernel");
}

// The last iteration's x += alpha p: the FP64 CG operator kernel applies an
// iteration's x update at the start of the next iteration (it holds p there
// anyway); the iteration that stopped the solve has no next one.
__global__ void x_finish_kernel(const double *x, const double *__restrict__ p, double *out, const CgState *st,
                                int64_t n) {
    const double alpha = st->alpha;
    for (int64_t l = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; l < n; l += int64_t(gridDim.x) * blockDim.x)
        out[l] = fma(alpha, p[l], x[l]);
}

int launch_x_finish(const Problem *P, double *out) {
    x_finish_kernel<<<stream_grid(P->nL), kThreads, 0, stream()>>>(P->x, P->p, out, P->st, P->nL);
    count_launches(1);
    return cuda_check(cudaGetLastError(), "x_finish_kernel");
}

// The update of solves of a given number of iterations: every copy of a node
// sums its copies in ascending order and updates itself, <r, r> in double-word
// FP32 per thread, 8 blocks per SM (E = 32^3, N = 7: 133 us, where owner rows
// take 78).
template <int NQ>
__global__ void __launch_bounds__(256) cg_update_class_kernel(double *__restrict__ r, const double *__restrict__ w,
                                                              int E, BoxDims bd, double *partials, int64_t cap,
                                                              CgState *st) {
    __shared__ double scratch[256];
    if (st->done) return;
    constexpr int V = UpdVec<NQ, double>::value;
    using RM = RowMap<NQ, V>;
    const double alpha = st->alpha;
    const int ntask = RM::tasks(E);
    const int lane = threadIdx.x & 31;
    const int nwarps = int(gridDim.x * blockDim.x) >> 5;
    DwAcc acc = acc_zero<DwAcc>();
    for (int task = int(blockIdx.x * blockDim.x + threadIdx.x) >> 5; task < ntask; task += nwarps) {
        const int l0 = RM::l0(task, lane, E);
        if (l0 >= 0) update_vec<NQ, V, double, DwAcc, true>(nullptr, r, nullptr, w, l0, bd, alpha, acc);
    }
    const double bs = block_sum_wide(acc_value(acc), scratch);
    double rho_new;
    if (grid_sum_groups(bs, partials, cap, &st->ticket_up, &rho_new) && threadIdx.x == 0) {
        cg_close_iteration(st, rho_new);
        if (!st->done && !dw_in_range(rho_new)) st->done = kDoneOutOfRange;
    }
}

template <int NQ>
static int launch_update_steps_nq(const Problem *P) {
    const int64_t tasks = RowMap<NQ, UpdVec<NQ, double>::value>::tasks(int(P->E));
    const int64_t blocks = std::min<int64_t>((tasks * 32 + 255) / 256, int64_t(sm_count()) * 8);
    cg_update_class_kernel<NQ><<<unsigned(blocks), 256, 0, stream()>>>(
        P->r, P->w, int(P->E), box_dims(P->nx, P->ny, P->nz), P->partials, P->partials_cap, P->st);
    count_launches(1);
    return cuda_check(cudaGetLastError(), "cg_update_class_kernel");
}

static int launch_update_steps(const Problem *P) {
    switch (P->nq) {
        case 2: return launch_update_steps_nq<2>(P);
        case 3: return launch_update_steps_nq<3>(P);
        case 4: return launch_update_steps_nq<4>(P);
        case 5: return launch_update_steps_nq<5>(P);
        case 6: return launch_update_steps_nq<6>(P);
        case 7: return launch_update_steps_nq<7>(P);
        case 8: return launch_update_steps_nq<8>(P);
        case 9: return launch_update_steps_nq<9>(P);
        case 10: return launch_update_steps_nq<10>(P);
        default: return set_error(SEM_EARG, "cg: unsupported order");
    }
}

int launch_cg_update(const Problem *P) {
    // <r, r> accumulated in double-word FP32 per thread (sem_box.cuh)
    return launch_update_rows<double>(P, P->r, P->w, P->st);
}

// Iterations per captured graph: the host polls the stop flag once per replay.
static int graph_iters_for(const Problem *P) {
    // small problems are launch-bound: more iterations per replay
    return P->nL < (1 << 20) ? 64 : 16;
}

static int capture_graph(Problem *P, bool steps) {
    if (P->graph_epoch != tune_epoch()) problem_drop_graphs(P);   // operator variant changed
    cudaGraphExec_t &graph = steps ? P->graph_steps : P->graph;
    if (graph) return SEM_OK;
    const int K = graph_iters_for(P);
    cudaGraph_t g = nullptr;
    int rc = cuda_check(cudaStreamBeginCapture(stream(), cudaStreamCaptureModeThreadLocal), "cg: begin capture");
    if (rc != SEM_OK) return rc;
    for (int k = 0; k < K && rc == SEM_OK; ++k) {
        rc = steps ? launch_ax_dw(P) : launch_ax_cg(P);
        if (rc == SEM_OK) rc = steps ? launch_update_steps(P) : launch_cg_update(P);
    }
    // launches inside a capture are counted at replay time instead
    count_launches(-2 * int64_t(K));
    const int rc_end = cuda_check(cudaStreamEndCapture(stream(), &g), "cg: end capture");
    if (rc == SEM_OK) rc = rc_end;
    if (rc == SEM_OK) rc = cuda_check(cudaGraphInstantiate(&graph, g, 0), "cg: instantiate");
    if (g) cudaGraphDestroy(g);
    if (rc == SEM_OK) {
        P->graph_iters = K;
        P->graph_stream = stream();
    }
    return rc;
}

int cg_solve(Problem *P, const double *b, double *x, double tol, int maxit, double *hist,
             int64_t *iters, double *rel_res) {
    if (maxit < 0) return set_error(SEM_EARG, "cg_solve: maxit must be >= 0");
    if (P->graph_stream != stream()) {
        problem_drop_graph(&P->graph);
        problem_drop_graph(&P->graph_steps);
    }
    // a given number of iterations: sem_ax_dw.cuh, where the table names the
    // fixed-point operator and the factors are within range
    int rc = SEM_OK;
    bool steps = !(tol > 0.0) && tune_get(kTuneF64, P->nq).variant == kAxLinesFX;
    if (steps) {
        rc = dw_prepare(P);
        steps = !P->dw_out;
    }
    if (rc == SEM_OK && !steps) rc = prepare_f64_variant(P);
    if (rc == SEM_OK) rc = launch_cg_init(P, b, maxit, tol, hist, steps);
    bool small = rc == SEM_OK && !steps && small_fits(P, false);
    if (rc == SEM_OK && !small) rc = capture_graph(P, steps);
    if (rc != SEM_OK) return rc;
    // at most maxit iterations are left to run; the flag stops earlier replays
    // short (a small problem's launches hold many more iterations than K)
    int64_t left = maxit;
    while (left > 0) {
        const int64_t K = small ? 1 : P->graph_iters;
        if (small) {
            bool refused = false;
            rc = launch_small(P, false, &refused);
            if (rc == SEM_OK && refused) {   // by the first launch, nothing has run
                small = false;
                rc = capture_graph(P, false);
                if (rc == SEM_OK) continue;
            }
        } else {
            rc = cuda_check(cudaGraphLaunch(steps ? P->graph_steps : P->graph, stream()), "cg: graph launch");
            if (rc == SEM_OK) count_launches(2 * K);
        }
        if (rc != SEM_OK) return rc;
        rc = cuda_check(cudaMemcpyAsync(P->st_host, P->st, sizeof(CgState), cudaMemcpyDeviceToHost, stream()),
                        "cg: state read");
        if (rc == SEM_OK)
            rc = cuda_check(cudaMemcpyAsync(status_host(), status_word(), sizeof(int32_t),
                                            cudaMemcpyDeviceToHost, stream()),
                            "cg: status read");
        if (rc != SEM_OK) return rc;
        rc = cuda_check(cudaStreamSynchronize(stream()), "cg: sync");
        if (rc != SEM_OK) return rc;
        if (*status_host() != 0) break;
        left -= K;
        if (P->st_host->done == kDoneOutOfRange) {
            // ||r|| left the range of double-word numbers: the general kernels
            // go on from this state
            steps = false;
            left = maxit - P->st_host->iter;
            rc = prepare_f64_variant(P);
            if (rc == SEM_OK) rc = capture_graph(P, false);
            if (rc == SEM_OK) rc = cuda_check(cudaMemsetAsync(&P->st->done, 0, sizeof(int32_t), stream()), "cg: resume");
            if (rc != SEM_OK) return rc;
        } else if (P->st_host->done) {
            break;
        }
    }
    rc = small ? cuda_check(cudaMemcpyAsync(x, P->x, sizeof(double) * P->nL, cudaMemcpyDeviceToDevice, stream()),
                            "cg: copy x")
               : launch_x_finish(P, x);
    if (rc == SEM_OK)
        rc = cuda_check(cudaMemcpyAsync(P->st_host, P->st, sizeof(CgState), cudaMemcpyDeviceToHost, stream()),
                        "cg: state read");
    if (rc == SEM_OK) rc = cuda_check(cudaStreamSynchronize(stream()), "cg: sync");
    if (rc != SEM_OK) return rc;
    rc = poll_status();
    if (rc != SEM_OK) return rc;
    *iters = P->st_host->iter;
    *rel_res = P->st_host->rho0 > 0.0 ? std::sqrt(P->st_host->rho / P->st_host->rho0) : 0.0;
    return SEM_OK;
}

}  // namespace sem
