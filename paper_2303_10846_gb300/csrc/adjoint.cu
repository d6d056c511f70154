// Host side of the adjoint ABI (include/rykov.h, "adjoint of the steady residual
// operator"): the second workspace, the steady residual, the vector-Jacobian product,
// the objectives and the restarted GMRES solve of (dR/dX)^T lam = -dJ/dX.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

#include "adjoint_dev.cuh"
#include "rykov_dev_fp64.cuh"
#include "rykov_ctx.h"

namespace rk {

constexpr int ADJ_WPB = 4;

struct AdjState {
    int gen = -1;                  // bind generation of the main workspace it belongs to
    int m = 0;                     // Krylov dimension of a restart cycle
    size_t np = 0, n = 0;          // padded / packed state-vector lengths
    double *f0 = nullptr, *fbar = nullptr, *nbg = nullptr, *tau = nullptr, *fpar = nullptr,
           *iterp = nullptr, *pout = nullptr, *part = nullptr, *hd = nullptr;
    // records of the state and sums of a product (AdjBufs, AdjArr), inverse micro diagonal
    double *fmom = nullptr, *fsum = nullptr, *csum = nullptr, *ceq = nullptr, *feq = nullptr, *fcoef = nullptr,
           *iD = nullptr;
    int* slot_mirg = nullptr;
    double* slot_AVn = nullptr;
    // padded state vectors [2 N Kp | 6 N | 6 N]
    double *vzero = nullptr, *jv = nullptr, *lam = nullptr, *rv = nullptr, *tmp = nullptr,
           *tmp2 = nullptr, *V = nullptr;
    double* stage = nullptr;       // packed staging for host inputs / outputs
    // macroscopic part of the preconditioner: a padded phi-block temporary, the
    // (W, q) outputs of the collision-coupling product, the macro adjoint iterate (by cell
    // and by colour position) and the constants and slots of its point updates
    double *pc1 = nullptr, *pcW = nullptr, *mY = nullptr, *mYp = nullptr, *mC = nullptr, *mS = nullptr;
    // mixed-precision contexts: FP64 copies of phi and of the frozen limiter values,
    // s_ij per slot (the FP64 view of the context's FP32 per-velocity arrays)
    double *phi64 = nullptr, *lstore64 = nullptr, *slot_s64 = nullptr;
    float* vf = nullptr;           // the phi block of v rounded to FP32
    double* hpin = nullptr;        // pinned host scratch
    int lam_obj = -1;              // objective of the stored lam (-1: none)
    long long lam_ver = -1;        // state version it was solved at
    long long launches = 0;
};

static inline int cdv(long long a, long long b) { return (int)((a + b - 1) / b); }

// out = -out on the phi block (the transposed sweeps' result), out = -in on (W, q)
__global__ void k_adj_precond_finish(const double* in, double* out, size_t n1, size_t np) {
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < np; t += (size_t)gridDim.x * blockDim.x)
        out[t] = t < n1 ? -out[t] : -in[t];
}

}  // namespace rk

using rk::AdjState;

void rk_adj_release(rk_ctx* ctx) {
    if (!ctx || !ctx->adj) return;
    if (ctx->adj->hpin) cudaFreeHost(ctx->adj->hpin);
    delete ctx->adj;
    ctx->adj = nullptr;
}

static size_t adj_carve(rk_ctx* ctx, int m, char* base, AdjState& A) {
    Carver cv{base};
    const size_t N = ctx->N, F = ctx->F, Kp = ctx->Kp, nnz = ctx->nnz, K = ctx->K;
    A.np = 2 * N * Kp + 12 * N;
    A.n = 2 * N * K + 12 * N;
    A.m = m;
    A.f0 = cv.take<double>(2 * F * Kp);
    A.fbar = cv.take<double>(2 * F * Kp);
    // shares of the neighbours: 2 ms per (cell, velocity), eight at least (the FP64 face
    // kernels of rk_steady_residual take their records here)
    size_t ms = 4;
    for (size_t i = 0; i < N; ++i) ms = std::max<size_t>(ms, ctx->slot_off[i + 1] - ctx->slot_off[i]);
    A.nbg = cv.take<double>(2 * ms * N * Kp);
    // and, between the products, the preconditioner's temporary and its input at the end of a
    // restart cycle (4 N K_pad + 12 N doubles of 8 N K_pad at least; each is written in full
    // before it is read)
    A.pc1 = A.nbg;
    A.tmp2 = A.nbg + 2 * N * Kp;
    A.fmom = cv.take<double>((size_t)rk::FMOM * (ctx->Fi + 1));
    A.fsum = cv.take<double>((size_t)(rk::ADJ_FS + 1) * (ctx->Fi + 1));
    A.feq = cv.take<double>((size_t)rk::EQA * (ctx->Fi + 1));
    A.fcoef = cv.take<double>((size_t)rk::ADJ_FC * (ctx->Fi + 1));
    A.csum = cv.take<double>((size_t)rk::ADJ_CS * N);
    A.ceq = cv.take<double>((size_t)rk::EQA * N);
    A.iD = cv.take<double>(N * Kp);
    A.slot_mirg = cv.take<int>(nnz);
    A.slot_AVn = cv.take<double>(nnz);
    A.tau = cv.take<double>(N);
    A.fpar = cv.take<double>((size_t)rk::ADJ_FPAR * (ctx->Fb + 1));
    A.iterp = cv.take<double>(4);
    A.pout = cv.take<double>(16);
    A.part = cv.take<double>((size_t)rk::VEC_GRID * rk::GM_MAX);
    A.hd = cv.take<double>(3 * rk::GM_MAX + 8);
    A.vzero = cv.take<double>(A.np);
    A.jv = cv.take<double>(A.np);
    A.lam = cv.take<double>(A.np);
    A.rv = cv.take<double>(A.np);
    A.tmp = cv.take<double>(A.np);
    A.V = cv.take<double>((size_t)(m + 1) * A.np);
    A.stage = cv.take<double>(A.n);
    A.pcW = cv.take<double>(12 * N);
    A.mY = cv.take<double>(6 * N);
    A.mYp = cv.take<double>(8 * N);
    A.mC = cv.take<double>(8 * N);
    A.mS = cv.take<double>(5 * ms * N);
    A.slot_s64 = cv.take<double>(nnz);
    if (ctx->prec == RK_MIXED) {
        A.phi64 = cv.take<double>(2 * N * Kp);
        A.lstore64 = cv.take<double>(2 * N * Kp);
        A.vf = cv.take<float>(2 * N * Kp);
    }
    return cv.off + 256;
}

static int need_adj(rk_ctx* ctx, const char* who) {
    if (!ctx) return RK_EINVAL;
    if (!ctx->bound) return fail(ctx, RK_ESTATE, std::string(who) + ": bind a workspace first");
    if (!ctx->adj || ctx->adj->gen != ctx->bind_gen)
        return fail(ctx, RK_ESTATE, std::string(who) + ": bind an adjoint workspace first");
    if (!ctx->have_state) return fail(ctx, RK_ESTATE, std::string(who) + ": set a state first");
    return RK_OK;
}

extern "C" int rk_state_len(const rk_ctx* ctx, int64_t* n) {
    if (!ctx || !n) return RK_EINVAL;
    *n = 2 * ctx->N * ctx->K + 12 * ctx->N;
    return RK_OK;
}

extern "C" int rk_adjoint_workspace_size(rk_ctx* ctx, int32_t krylov_dim, size_t* bytes) {
    if (!ctx || !bytes) return RK_EINVAL;
    if (krylov_dim < 1 || krylov_dim > rk::GM_MAX)
        return fail(ctx, RK_EINVAL, "rk_adjoint_workspace_size: krylov_dim out of range");
    if (!ctx->mesh_ok || !ctx->dvs_ok) return fail(ctx, RK_ESTATE, "rk_adjoint_workspace_size: upload mesh and DVS first");
    AdjState A;
    *bytes = adj_carve(ctx, krylov_dim, nullptr, A);
    return RK_OK;
}

extern "C" int rk_bind_adjoint_workspace(rk_ctx* ctx, int32_t krylov_dim, void* dev_ptr, size_t bytes) {
    if (!ctx || !dev_ptr) return RK_EINVAL;
    if (!ctx->bound) return fail(ctx, RK_ESTATE, "rk_bind_adjoint_workspace: bind the main workspace first");
    size_t need = 0;
    int rc = rk_adjoint_workspace_size(ctx, krylov_dim, &need);
    if (rc) return rc;
    if (bytes < need)
        return fail(ctx, RK_ENOMEM, "rk_bind_adjoint_workspace: workspace too small (" + std::to_string(bytes) +
                                        " < " + std::to_string(need) + ")");
    if (reinterpret_cast<uintptr_t>(dev_ptr) & 255)
        return fail(ctx, RK_EINVAL, "rk_bind_adjoint_workspace: pointer not 256-byte aligned");
    rk_adj_release(ctx);
    AdjState* A = new (std::nothrow) AdjState();
    if (!A) return fail(ctx, RK_ENOMEM, "rk_bind_adjoint_workspace: host allocation failed");
    if (cudaMallocHost(&A->hpin, (3 * rk::GM_MAX + 16) * sizeof(double)) != cudaSuccess) {
        delete A;
        return fail(ctx, RK_ECUDA, "rk_bind_adjoint_workspace: pinned host buffer");
    }
    ctx->adj = A;
    adj_carve(ctx, krylov_dim, static_cast<char*>(dev_ptr), *A);
    cudaStream_t s = ctx->stream;
    const size_t N = ctx->N, nnz = ctx->nnz;
    // mirror slots (the same face in the neighbour's list) and A_f / V_neighbour
    std::vector<int> mir(nnz, -1);
    std::vector<double> avn(nnz, 0.0);
    for (size_t i = 0; i < N; ++i) {
        for (int m = ctx->slot_off[i]; m < ctx->slot_off[i + 1]; ++m) {
            const int j = ctx->slot_nbr[m];
            if (j < 0) continue;
            for (int mm = ctx->slot_off[j]; mm < ctx->slot_off[j + 1]; ++mm)
                if (ctx->slot_face[mm] == ctx->slot_face[m]) mir[m] = mm;
            avn[m] = ctx->fa[ctx->slot_face[m]] / ctx->cv[j];
        }
    }
    // zero everything once: the K padding of every vector stays 0
    CK(cudaMemsetAsync(dev_ptr, 0, need - 256, s));
    CK(cudaMemcpyAsync(A->slot_mirg, mir.data(), nnz * sizeof(int), cudaMemcpyHostToDevice, s));
    CK(cudaMemcpyAsync(A->slot_AVn, avn.data(), nnz * sizeof(double), cudaMemcpyHostToDevice, s));
    {
        const rk::DevBase& b = ctx->prec == RK_FP64 ? static_cast<const rk::DevBase&>(ctx->dd)
                                                    : static_cast<const rk::DevBase&>(ctx->df);
        rk::k_adj_slot_s<<<rk::cdv(nnz, 256), 256, 0, s>>>(b, A->slot_s64);
        CK(cudaGetLastError());
    }
    CK(cudaStreamSynchronize(s));
    A->gen = ctx->bind_gen;
    return RK_OK;
}

// The FP64 view of the context: the FP64 context's own arrays, or, for a mixed
// context, its FP64 geometry and state with FP64 copies of the per-velocity arrays
static rk::Dev<double> dview(rk_ctx* ctx, AdjState& A) {
    if (ctx->prec == RK_FP64) return ctx->dd;
    rk::Dev<double> d{};
    static_cast<rk::DevBase&>(d) = static_cast<const rk::DevBase&>(ctx->df);
    const double v[8] = {d.R, d.Z, d.mu_ref, d.T_ref, d.omega_vis, d.omega0, d.omega1, d.delta};
    for (int j = 0; j < 8; ++j) d.tp[j] = v[j];
    d.slot_nT = const_cast<double*>(d.slot_n);
    d.slot_AVT = d.slot_AV;
    d.slot_dT = d.slot_d;
    d.slot_lsqT = d.slot_lsq;
    d.slot_sT = A.slot_s64;
    d.fnT = const_cast<double*>(d.fn);
    d.fsT = d.fs;
    d.uT = d.u;
    d.wT = d.w;
    d.phi = A.phi64;
    d.face = A.fbar;
    d.res = d.dphi = nullptr;
    d.lstore = A.lstore64;
    d.debug = 0;
    return d;
}

// mixed contexts: refresh the FP64 copies of phi and of the frozen limiter values
static cudaError_t adj_sync(rk_ctx* ctx, AdjState& A) {
    if (ctx->prec != RK_MIXED) return cudaSuccess;
    const size_t n = 2 * (size_t)ctx->N * ctx->Kp;
    rk::k_adj_upcast<<<1216, 256, 0, ctx->stream>>>(ctx->df.phi, A.phi64, n);
    rk::k_adj_upcast<<<1216, 256, 0, ctx->stream>>>(ctx->df.lstore, A.lstore64, n);
    A.launches += 2;
    return cudaGetLastError();
}

// Per-velocity arithmetic of the adjoint kernels: FP64 for FP64 contexts; FP32 with
// compensated velocity sums for mixed-precision contexts (the state and the vectors
// stay FP64), unless RYKOV_ADJ_FP64=1 asks for FP64 arithmetic there too
static bool adj_fp32(const rk_ctx* ctx) {
    if (ctx->prec != RK_MIXED) return false;
    const char* v = std::getenv("RYKOV_ADJ_FP64");
    return !(v && std::strcmp(v, "0") != 0);
}

// ---- kernel sequences -------------------------------------------------------------
static rk::AdjBufs adj_bufs(rk_ctx* ctx, AdjState& A, const double* v, double* o) {
    rk::AdjBufs a{};
    const size_t N = ctx->N, n1 = 2 * N * (size_t)ctx->Kp;
    a.vW = v + n1; a.vq = v + n1 + 6 * N;
    a.ophi = o; a.oW = o + n1; a.oq = o + n1 + 6 * N;
    a.slot_mirg = A.slot_mirg; a.slot_AVn = A.slot_AVn;
    a.tau = A.tau; a.fpar = A.fpar; a.iterp = A.iterp;
    a.fmom = A.fmom; a.fsum = A.fsum; a.csum = A.csum;
    a.obj_scale = 0.0; a.objective = 0;
    a.edrag[0] = 1.0; a.edrag[1] = a.edrag[2] = 0.0;
    for (int b = 0; b < MAX_BC; ++b) {
        if (ctx->bck[b] != RK_FARFIELD) continue;
        const double* U = ctx->bcv + 5 * b + 1;
        const double nrm = std::sqrt(U[0] * U[0] + U[1] * U[1] + U[2] * U[2]);
        if (nrm > 0.0) {
            for (int d = 0; d < 3; ++d) a.edrag[d] = U[d] / nrm;
        }
        break;
    }
    return a;
}

// the arrays in the arithmetic type; v: the phi block of the vector (FP64: the vector
// itself; FP32: A.vf), o: the output vector (FP64: the cell terms go there directly)
template <typename S>
static rk::AdjArr<S> adj_arr(rk_ctx* ctx, AdjState& A, const rk::Dev<double>& d, const double* v, double* o) {
    rk::AdjArr<S> r{};
    const size_t FK2 = 2 * (size_t)ctx->F * ctx->Kp;
    if constexpr (sizeof(S) == 4) {
        r.u = ctx->df.uT; r.w = ctx->df.wT; r.phi = ctx->df.phi; r.f0 = ctx->df.face;
        r.lstore = ctx->df.lstore;
        r.v = A.vf;
        // fbar in the lower half of its buffer, the cell terms (F >= N) in the upper
        r.oc = reinterpret_cast<float*>(A.fbar) + FK2;
    } else {
        r.u = d.u; r.w = d.w; r.phi = d.phi; r.f0 = A.f0;
        r.lstore = d.lstore;
        r.v = v;
        r.oc = o;
    }
    r.fbar = reinterpret_cast<S*>(A.fbar);
    r.nb = reinterpret_cast<S*>(A.nbg);
    r.iD = reinterpret_cast<S*>(A.iD);
    r.ceq = reinterpret_cast<S*>(A.ceq);
    r.feq = reinterpret_cast<S*>(A.feq);
    r.fcoef = reinterpret_cast<S*>(A.fcoef);
    return r;
}

// What depends on the state alone: the limited reconstruction phi(x_f - u s), tau(W), and
// the equilibrium constants of cells and interior faces
template <typename S>
static cudaError_t adj_prepare_t(rk_ctx* ctx, AdjState& A) {
    cudaStream_t s = ctx->stream;
    rk::Dev<double> d = dview(ctx, A);
    d.iterp = A.iterp;
    if constexpr (sizeof(S) == 4) {
        // the context's own FP32 reconstruction, written to its face array (scratch of the
        // iteration: the rows are no finished faces afterwards)
        rk::Dev<float> df = ctx->df;
        df.iterp = A.iterp;
        cudaError_t e = rk::Launch<float>::recon(df, s, ctx->prof);
        if (e != cudaSuccess) return e;
        ctx->faces_partial = ctx->faces_redo = true;
    } else {
        d.face = A.f0;
        rk::launch_recon_d<false>(d, s, nullptr, (int)ctx->N);
    }
    const rk::AdjBufs a = adj_bufs(ctx, A, A.vzero, A.tmp);
    const rk::AdjArr<S> r = adj_arr<S>(ctx, A, d, A.vzero, A.tmp);
    rk::k_adj_cstate<S><<<rk::cdv(ctx->N, 64), 64, 0, s>>>(d, A.tau, r.ceq);
    if (ctx->Fi) {
        constexpr int W = rk::ADJ_WPB;
        rk::k_adj_mom<W, S><<<rk::cdv(ctx->Fi, W), W * 32, 0, s>>>(d, a, r);
        rk::k_adj_fstate<S><<<rk::cdv(ctx->Fi, 64), 64, 0, s>>>(d, a, r);
    }
    A.launches += 4;
    return cudaGetLastError();
}
static cudaError_t adj_mode(rk_ctx* ctx, AdjState& A) {
    // the steady operator's reconstruction: the limiter of rk_params, with the stored
    // values once the iteration has frozen them
    double mode = (double)ctx->p.limiter;
    if (ctx->p.limiter == 1 && ctx->p.limiter_freeze > 0 && ctx->iter >= ctx->p.limiter_freeze) mode = 3.0;
    const double ip[4] = {0.0, mode, 0.0, 0.0};
    return cudaMemcpyAsync(A.iterp, ip, sizeof(ip), cudaMemcpyHostToDevice, ctx->stream);
}
static cudaError_t adj_prepare(rk_ctx* ctx, AdjState& A) {
    cudaError_t e = adj_mode(ctx, A);
    if (e != cudaSuccess) return e;
    if (adj_fp32(ctx)) return adj_prepare_t<float>(ctx, A);
    if ((e = adj_sync(ctx, A)) != cudaSuccess) return e;
    return adj_prepare_t<double>(ctx, A);
}

template <int W, typename S>
static void adj_gather(const rk::Dev<double>& d, const rk::AdjBufs& a, const rk::AdjArr<S>& r, cudaStream_t s) {
    const int g = rk::cdv(d.N, W);
    if (d.ms <= 4) rk::k_adj_gather<W, S, 4><<<g, W * 32, 0, s>>>(d, a, r);
    else if (d.ms <= 6) rk::k_adj_gather<W, S, 6><<<g, W * 32, 0, s>>>(d, a, r);
    else rk::k_adj_gather<W, S, 8><<<g, W * 32, 0, s>>>(d, a, r);
}

// o = (dR/dX)^T v (padded vectors), pout = (dR/dp)^T v.  v null: v = 0, for which only the
// boundary faces' seeds and the gathers are run: with obj_scale = 1 that gives dJ/dX,
// pout[0-5] = dJ/dp|_X, pout[6] = J, pout[7-9] = force.  src: A.vf holds the phi block
// of v already, whose FP64 phi block is then that of src (the packed vector), which may be
// dst: the last kernel alone writes there.  dst, ld: where the phi block of the result goes
// (rows of ld doubles).
template <typename S>
static cudaError_t adj_apply_t(rk_ctx* ctx, AdjState& A, const double* v, double* o, double obj_scale, int objective,
                               const double* src, double* dst, int ld) {
    constexpr int W = rk::ADJ_WPB;
    const bool zero = v == nullptr, have_vf = src != nullptr;
    if (zero) v = A.vzero;
    const size_t N = ctx->N, NK2 = 2 * N * (size_t)ctx->Kp;
    rk::AdjBufs a = adj_bufs(ctx, A, v, o);
    a.obj_scale = obj_scale;
    a.objective = objective;
    const rk::Dev<double> d = dview(ctx, A);
    const rk::AdjArr<S> r = adj_arr<S>(ctx, A, d, v, o);
    cudaStream_t s = ctx->stream;
    const int gc = rk::cdv(ctx->N, W);
    cudaError_t e = cudaSuccess;
    if (sizeof(S) == 4 && zero) {
        if ((e = cudaMemsetAsync(A.vf, 0, NK2 * sizeof(float), s)) != cudaSuccess) return e;
    } else if (sizeof(S) == 4 && !have_vf) {
        rk::k_adj_downcast<<<1216, 256, 0, s>>>(v, A.vf, NK2);
        A.launches++;
    }
    if (zero) {
        if ((e = cudaMemsetAsync(r.oc, 0, NK2 * sizeof(S), s)) != cudaSuccess) return e;
        if ((e = cudaMemsetAsync(a.oW, 0, 12 * N * sizeof(double), s)) != cudaSuccess) return e;
        if ((e = cudaMemsetAsync(r.fbar, 0, 2 * (size_t)ctx->F * ctx->Kp * sizeof(S), s)) != cudaSuccess) return e;
    } else {
        rk::k_adj_cell<W, S, true, false><<<gc, W * 32, 0, s>>>(d, a, r);
        rk::k_adj_crev<S><<<rk::cdv(ctx->N, 64), 64, 0, s>>>(d, a);
        A.launches += 2;
        if (ctx->Fi) {
            const int gf = rk::cdv(ctx->Fi, W);
            rk::k_adj_face_a<W, S><<<gf, W * 32, 0, s>>>(d, a, r);
            rk::k_adj_frev<S><<<rk::cdv(ctx->Fi, 64), 64, 0, s>>>(d, a, r);
            rk::k_adj_face_b<W, S><<<gf, W * 32, 0, s>>>(d, a, r);
            A.launches += 3;
        }
    }
    if (ctx->Fb) {
        rk::k_adj_face_boundary<128, S><<<ctx->Fb, 128, 0, s>>>(d, a, r, have_vf ? src : v, have_vf ? (int)ctx->K : ctx->Kp);
        rk::k_adj_params<<<1, 320, 0, s>>>(A.fpar, ctx->Fb, A.pout);
        A.launches += 2;
    } else if ((e = cudaMemsetAsync(A.pout, 0, 16 * sizeof(double), s)) != cudaSuccess) {
        return e;
    }
    adj_gather<W, S>(d, a, r, s);
    rk::k_adj_gather2<W, S><<<gc, W * 32, 0, s>>>(d, a, r, dst, ld);
    A.launches += 2;
    return cudaGetLastError();
}
static cudaError_t adj_apply(rk_ctx* ctx, AdjState& A, const double* v, double* o, double obj_scale, int objective) {
    return adj_fp32(ctx) ? adj_apply_t<float>(ctx, A, v, o, obj_scale, objective, nullptr, o, ctx->Kp)
                         : adj_apply_t<double>(ctx, A, v, o, obj_scale, objective, nullptr, o, ctx->Kp);
}

// What the preconditioner needs of the state: the inverse micro diagonal and the constants
// of the transposed macro updates.  Once per solve.  Its spectral radii are the last
// iteration's, one step behind the state that it left, or W's for any other state (they
// enter the preconditioner alone, so a solve that reaches its tolerance does not depend on
// them; one that stops at max_iter does).
template <typename S>
static cudaError_t adj_pc_prepare_t(rk_ctx* ctx, AdjState& A) {
    const rk::Dev<double> d = dview(ctx, A);
    const rk::AdjBufs a = adj_bufs(ctx, A, A.vzero, A.tmp);
    const rk::AdjArr<S> r = adj_arr<S>(ctx, A, d, A.vzero, A.tmp);
    constexpr int W = rk::ADJ_WPB;
    rk::k_adj_sweep<W, S, true><<<rk::cdv(ctx->N, W), W * 32, 0, ctx->stream>>>(d, a, r, nullptr, (int)ctx->N, nullptr, nullptr);
    if (!ctx->have_radii) {
        rk::k_face_radius<double><<<rk::cdv(ctx->F, 64), 64, 0, ctx->stream>>>(d);
        A.launches++;
    }
    rk::k_adj_macro_prep<<<rk::cdv(ctx->N, 128), 128, 0, ctx->stream>>>(d, ctx->sched.col_cell, A.tau, A.mC, A.mS);
    A.launches += 2;
    return cudaGetLastError();
}
static cudaError_t adj_pc_prepare(rk_ctx* ctx, AdjState& A) {
    return adj_fp32(ctx) ? adj_pc_prepare_t<float>(ctx, A) : adj_pc_prepare_t<double>(ctx, A);
}

// The transposed micro sweeps of r into y.  A repeated phase (the turn of a sweep) leaves
// y as it is, the update of a cell depending on its neighbours alone: each is done once.
template <typename S>
static void adj_micro_sweeps(rk_ctx* ctx, AdjState& A, const rk::Dev<double>& d, const rk::AdjBufs& a,
                             const double* b, double* y) {
    constexpr int W = rk::ADJ_WPB;
    const rk::AdjArr<S> r = adj_arr<S>(ctx, A, d, b, y);
    for (const rk::Phase& ph : rk::sgs_phases(ctx->sched, ctx->p.n_micro_sgs)) {
        const int lo = ctx->col_off[ph.col], n = ctx->col_off[ph.col + 1] - lo;
        rk::k_adj_sweep<W, S, false><<<rk::cdv(n, W), W * 32, 0, ctx->stream>>>(d, a, r, ctx->sched.col_cell + lo, n, b, y);
        A.launches++;
    }
}

// out = P^-1 in: transposed colour sweeps on the phi block (negated), -in on (W, q)
static cudaError_t adj_precond(rk_ctx* ctx, AdjState& A, const double* in, double* out) {
    cudaStream_t s = ctx->stream;
    const size_t n1 = 2 * (size_t)ctx->N * ctx->Kp;
    cudaError_t e = cudaMemsetAsync(out, 0, n1 * sizeof(double), s);
    if (e != cudaSuccess) return e;
    const rk::AdjBufs a = adj_bufs(ctx, A, in, out);
    const rk::Dev<double> d = dview(ctx, A);
    if (adj_fp32(ctx)) adj_micro_sweeps<float>(ctx, A, d, a, in, out);
    else adj_micro_sweeps<double>(ctx, A, d, a, in, out);
    rk::k_adj_precond_finish<<<1216, 256, 0, s>>>(in, out, n1, A.np);
    A.launches++;
    return cudaGetLastError();
}

// out = P^-T in with the macroscopic coupling of the forward iteration (transposed):
//   t     = S^-T (in_phi + M_Y^T in_Y)              transposed micro sweeps
//   x     = L^-T (B_W^T t)                          transposed macro PR-SGS sweeps
//   out   = -(t + M_W^T x),  -in_Y                  (the sign convention of adj_precond)
template <typename S>
static cudaError_t adj_precond_macro(rk_ctx* ctx, AdjState& A, const double* in, double* out) {
    cudaStream_t s = ctx->stream;
    constexpr int W = rk::ADJ_WPB;
    const size_t N = ctx->N, n1 = 2 * N * (size_t)ctx->Kp;
    const rk::Dev<double> d = dview(ctx, A);
    rk::k_adj_momT<<<rk::cdv(ctx->N, 4), 128, 0, s>>>(d, in, in + n1, in + n1 + 6 * N, A.pc1);
    cudaError_t e = cudaMemsetAsync(out, 0, n1 * sizeof(double), s);
    if (e != cudaSuccess) return e;
    const rk::AdjBufs a = adj_bufs(ctx, A, in, out);
    adj_micro_sweeps<S>(ctx, A, d, a, A.pc1, out);
    // B_W^T t: the collision coupling's W derivative applied to t (zero (W, q) weights)
    rk::AdjBufs b = adj_bufs(ctx, A, out, nullptr);
    b.vW = A.vzero + n1;
    b.vq = b.vW + 6 * N;
    b.oW = A.pcW;
    b.oq = A.pcW + 6 * N;
    if (sizeof(S) == 4) {
        rk::k_adj_downcast<<<1216, 256, 0, s>>>(out, A.vf, n1);
        A.launches++;
    }
    rk::k_adj_cell<W, S, false, true><<<rk::cdv(ctx->N, W), W * 32, 0, s>>>(d, b, adj_arr<S>(ctx, A, d, out, nullptr));
    rk::k_adj_crev<S><<<rk::cdv(ctx->N, 64), 64, 0, s>>>(d, b);
    // L^-T (B_W^T t) by transposed colour sweeps of the macro operator, each phase launched
    // ahead of its turn (programmatic serialisation) but the first
    if ((e = cudaMemsetAsync(A.mYp, 0, 8 * N * sizeof(double), s)) != cudaSuccess) return e;
    const rk::DevBase& db = d;
    bool first = true;
    for (const rk::Phase& ph : rk::sgs_phases(ctx->sched, ctx->p.n_macro_sgs)) {
        const int lo = ctx->col_off[ph.col], n = ctx->col_off[ph.col + 1] - lo, L = rk::macro_lanes(n, d.ms);
        e = rk::launch_phase(L == 1 ? rk::k_adj_macro_sweepT<1> : L == 2 ? rk::k_adj_macro_sweepT<2>
                             : L == 4 ? rk::k_adj_macro_sweepT<4> : rk::k_adj_macro_sweepT<8>,
                             (long long)n * L, !first, s, db, ctx->sched.col_cell, lo, n, A.mC, A.mS, A.pcW, A.mYp);
        if (e != cudaSuccess) return e;
        first = false;
        A.launches++;
    }
    rk::k_adj_macro_out<<<rk::cdv(ctx->N, 128), 128, 0, s>>>(db, A.mYp, A.mY);
    // t + M_W^T x, then the signs
    rk::k_adj_momT<<<rk::cdv(ctx->N, 4), 128, 0, s>>>(d, out, A.mY, nullptr, out);
    rk::k_adj_precond_finish<<<1216, 256, 0, s>>>(in, out, n1, A.np);
    A.launches += 6;
    return cudaGetLastError();
}

// the preconditioner of the adjoint solve: with the macroscopic coupling (default), or
// the transposed micro sweeps alone (RYKOV_ADJ_PC=micro)
static cudaError_t adj_pc(rk_ctx* ctx, AdjState& A, const double* in, double* out) {
    const char* v = std::getenv("RYKOV_ADJ_PC");
    if (v && std::strcmp(v, "micro") == 0) return adj_precond(ctx, A, in, out);
    return adj_fp32(ctx) ? adj_precond_macro<float>(ctx, A, in, out) : adj_precond_macro<double>(ctx, A, in, out);
}

// dots of x with V_0..V_{m-1} into dev (device), deterministic
static void adj_mdot(rk_ctx* ctx, AdjState& A, const double* x, const double* V, int m, double* dev) {
    rk::k_vec_mdot<<<rk::VEC_GRID, rk::VEC_BS, 0, ctx->stream>>>(x, V, A.np, m, A.np, A.part);
    rk::k_vec_finish<<<m, 32, 0, ctx->stream>>>(A.part, m, dev);
    A.launches += 2;
}

static int adj_norm(rk_ctx* ctx, AdjState& A, const double* x, double* out) {
    adj_mdot(ctx, A, x, x, 1, A.hd + 3 * rk::GM_MAX);
    CK(cudaMemcpyAsync(A.hpin, A.hd + 3 * rk::GM_MAX, sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    *out = std::sqrt(A.hpin[0]);
    return RK_OK;
}

static void vec_axpby(rk_ctx* ctx, AdjState& A, double a, const double* x, double b, double* y) {
    rk::k_vec_axpby<<<1216, 256, 0, ctx->stream>>>(a, x, b, y, A.np);
    A.launches++;
}

// packed <-> padded: the phi rows by a kernel, the W and q blocks as they are.  vec is
// the padded vector; phi (of type S) is where its phi block goes to or comes from
template <typename S>
static cudaError_t adj_unpack(rk_ctx* ctx, AdjState& A, const double* x, S* phi, double* vec) {
    const size_t N = ctx->N, rows = 2 * N, n1 = rows * (size_t)ctx->Kp, k1 = rows * (size_t)ctx->K;
    rk::k_adj_unpack<S><<<rk::cdv(rows, 8), 256, 0, ctx->stream>>>(x, rows, (int)ctx->K, ctx->Kp, phi);
    A.launches++;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return cudaMemcpyAsync(vec + n1, x + k1, 12 * N * sizeof(double), cudaMemcpyDeviceToDevice, ctx->stream);
}
template <typename S>
static cudaError_t adj_pack(rk_ctx* ctx, AdjState& A, const S* phi, const double* W, const double* q, double* x) {
    const size_t N = ctx->N, rows = 2 * N, k1 = rows * (size_t)ctx->K;
    if (phi) {
        rk::k_adj_pack<S><<<rk::cdv(rows, 8), 256, 0, ctx->stream>>>(phi, rows, (int)ctx->K, ctx->Kp, x);
        A.launches++;
    }
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(x + k1, W, 6 * N * sizeof(double), cudaMemcpyDeviceToDevice, ctx->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(x + k1 + 6 * N, q, 6 * N * sizeof(double), cudaMemcpyDeviceToDevice, ctx->stream);
    return e;
}
// packed device vector x -> the caller's (device: already there); synchronises
static int give_vec(rk_ctx* ctx, AdjState& A, const double* x, double* out, int on_device) {
    if (!on_device) CK(cudaMemcpyAsync(out, x, A.n * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    return RK_OK;
}
// padded device vector -> packed output (host or device); synchronises
static int store_vec(rk_ctx* ctx, AdjState& A, const double* vec, double* x, int on_device) {
    const size_t N = ctx->N, n1 = 2 * N * (size_t)ctx->Kp;
    double* to = on_device ? x : A.stage;
    CK(adj_pack(ctx, A, vec, vec + n1, vec + n1 + 6 * N, to));
    return give_vec(ctx, A, to, x, on_device);
}

// ---- ABI --------------------------------------------------------------------------
extern "C" int rk_get_state(rk_ctx* ctx, double* x, int on_device) {
    int rc = need_adj(ctx, "rk_get_state");
    if (rc) return rc;
    if (!x) return fail(ctx, RK_EINVAL, "rk_get_state: null pointer");
    AdjState& A = *ctx->adj;
    double* to = on_device ? x : A.stage;
    if (ctx->prec == RK_FP64) CK(adj_pack(ctx, A, ctx->dd.phi, ctx->dd.W, ctx->dd.q, to));
    else CK(adj_pack(ctx, A, ctx->df.phi, ctx->df.W, ctx->df.q, to));
    return give_vec(ctx, A, to, x, on_device);
}

extern "C" int rk_put_state(rk_ctx* ctx, const double* x, int on_device) {
    if (!ctx) return RK_EINVAL;
    if (!ctx->adj || ctx->adj->gen != ctx->bind_gen || !ctx->bound)
        return fail(ctx, RK_ESTATE, "rk_put_state: bind the workspaces first");
    if (!x) return fail(ctx, RK_EINVAL, "rk_put_state: null pointer");
    AdjState& A = *ctx->adj;
    const size_t N = ctx->N, rows = 2 * N, k1 = rows * (size_t)ctx->K;
    const double* src = x;
    if (!on_device) {
        CK(cudaMemcpyAsync(A.stage, x, A.n * sizeof(double), cudaMemcpyHostToDevice, ctx->stream));
        src = A.stage;
    }
    // a mixed context stores phi in FP32 (rounded)
    if (ctx->prec == RK_FP64)
        rk::k_adj_unpack<double><<<rk::cdv(rows, 8), 256, 0, ctx->stream>>>(src, rows, (int)ctx->K, ctx->Kp, ctx->dd.phi);
    else
        rk::k_adj_unpack<float><<<rk::cdv(rows, 8), 256, 0, ctx->stream>>>(src, rows, (int)ctx->K, ctx->Kp, ctx->df.phi);
    CK(cudaGetLastError());
    const rk::DevBase& d = ctx->prec == RK_FP64 ? static_cast<const rk::DevBase&>(ctx->dd)
                                                : static_cast<const rk::DevBase&>(ctx->df);
    // the last iteration's radii stay with the state that it left; another W has its own
    if (ctx->have_radii) {
        int* differ = reinterpret_cast<int*>(A.hd);
        CK(cudaMemsetAsync(differ, 0, sizeof(int), ctx->stream));
        rk::k_adj_differ<<<rk::cdv(6 * N, 256), 256, 0, ctx->stream>>>(src + k1, d.W, 6 * N, differ);
        CK(cudaGetLastError());
        CK(cudaMemcpyAsync(A.hpin, differ, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    }
    CK(cudaMemcpyAsync(d.W, src + k1, 6 * N * sizeof(double), cudaMemcpyDeviceToDevice, ctx->stream));
    CK(cudaMemcpyAsync(d.q, src + k1 + 6 * N, 6 * N * sizeof(double), cudaMemcpyDeviceToDevice, ctx->stream));
    CK(cudaMemsetAsync(d.iterp, 0, 4 * sizeof(double), ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    if (ctx->have_radii) {
        int differ = 0;
        std::memcpy(&differ, A.hpin, sizeof(int));
        ctx->have_radii = differ == 0;
    }
    ctx->iter = 0;
    ctx->have_state = true;
    ctx->state_ver++;
    return RK_OK;
}

extern "C" int rk_steady_residual(rk_ctx* ctx, double* r, int on_device) {
    int rc = need_adj(ctx, "rk_steady_residual");
    if (rc) return rc;
    if (!r) return fail(ctx, RK_EINVAL, "rk_steady_residual: null pointer");
    AdjState& A = *ctx->adj;
    CK(adj_mode(ctx, A));
    CK(adj_sync(ctx, A));
    // forward face pass of the steady operator into the fbar scratch (FP64)
    rk::Dev<double> d = dview(ctx, A);
    d.iterp = A.iterp;
    d.face = A.fbar;
    d.debug = 0;
    cudaStream_t s = ctx->stream;
    rk::launch_recon_d<false>(d, s, nullptr, (int)ctx->N);
    if (ctx->prec == RK_MIXED) {
        // scratch of the FP64 face kernels (44 doubles a face, at most 4 N interior faces)
        // and |u|^2/2 in the gradient-adjoint buffer (256 N doubles at least), not in use here
        d.fmom = A.nbg;
        d.feq = d.fmom + (size_t)rk::FMOM * (ctx->Fi + 1);
        double* u2 = d.feq + (size_t)rk::FEQ * (ctx->Fi + 1);
        rk::k_adj_u2<<<rk::cdv(ctx->Kp, 128), 128, 0, s>>>(d, u2);
        d.u2h = u2;
        A.launches++;
    }
    if (ctx->Fi) rk::launch_faces_d(d, s);
    if (ctx->Fb) rk::k_face_boundary<double, 128><<<ctx->Fb, 128, 0, s>>>(d, nullptr);
    rk::AdjBufs a = adj_bufs(ctx, A, A.vzero, A.tmp);
    rk::k_adj_residual<rk::ADJ_WPB><<<rk::cdv(ctx->N, rk::ADJ_WPB), rk::ADJ_WPB * 32, 0, s>>>(d, a);
    A.launches += 4;
    CK(cudaGetLastError());
    return store_vec(ctx, A, A.tmp, r, on_device);
}

extern "C" int rk_vjp(rk_ctx* ctx, const double* v, double* out, double* out_params, int on_device) {
    int rc = need_adj(ctx, "rk_vjp");
    if (rc) return rc;
    if (!v || !out) return fail(ctx, RK_EINVAL, "rk_vjp: null pointer");
    AdjState& A = *ctx->adj;
    const size_t N = ctx->N, n1 = 2 * N * (size_t)ctx->Kp;
    const double* src = v;
    if (!on_device) {
        CK(cudaMemcpyAsync(A.stage, v, A.n * sizeof(double), cudaMemcpyHostToDevice, ctx->stream));
        src = A.stage;
    }
    // the result's phi rows go to the packed output directly.  A host call reuses the staging
    // vector, and an output over the input v is fine too: v has been unpacked by then
    double* to = on_device ? out : A.stage;
    if (adj_fp32(ctx)) {
        CK(adj_unpack(ctx, A, src, A.vf, A.rv));
        CK(adj_prepare(ctx, A));
        CK(adj_apply_t<float>(ctx, A, A.rv, A.tmp, 0.0, 0, src, to, (int)ctx->K));
    } else {
        CK(adj_unpack(ctx, A, src, A.rv, A.rv));
        CK(adj_prepare(ctx, A));
        CK(adj_apply_t<double>(ctx, A, A.rv, A.tmp, 0.0, 0, nullptr, to, (int)ctx->K));
    }
    CK(adj_pack(ctx, A, (const double*)nullptr, A.tmp + n1, A.tmp + n1 + 6 * N, to));
    if (out_params) CK(cudaMemcpyAsync(A.hpin, A.pout, 6 * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    if ((rc = give_vec(ctx, A, to, out, on_device))) return rc;
    if (out_params) std::memcpy(out_params, A.hpin, 6 * sizeof(double));
    return RK_OK;
}

// J, force and dJ/dp|_X (host), dJ/dX into A.jv; drag adds the explicit dependence of
// e = U_inf / |U_inf| on the farfield velocity
static int objective_impl(rk_ctx* ctx, AdjState& A, int objective, double* J, double dJdp[6]) {
    CK(adj_prepare(ctx, A));
    CK(adj_apply(ctx, A, nullptr, A.jv, 1.0, objective));
    CK(cudaMemcpyAsync(A.hpin, A.pout, 10 * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    for (int j = 0; j < 6; ++j) dJdp[j] = A.hpin[j];
    *J = A.hpin[6];
    if (objective == RK_OBJ_DRAG) {
        for (int b = 0; b < MAX_BC; ++b) {
            if (ctx->bck[b] != RK_FARFIELD) continue;
            const double* U = ctx->bcv + 5 * b + 1;
            const double nrm = std::sqrt(U[0] * U[0] + U[1] * U[1] + U[2] * U[2]);
            if (nrm > 0.0) {
                const double* Fo = A.hpin + 7;
                const double Fe = (Fo[0] * U[0] + Fo[1] * U[1] + Fo[2] * U[2]) / nrm;
                for (int d = 0; d < 3; ++d) dJdp[2 + d] += (Fo[d] - Fe * U[d] / nrm) / nrm;
            }
            break;
        }
    }
    return RK_OK;
}

extern "C" int rk_objective(rk_ctx* ctx, int objective, double* J, double* dJdX, double* dJdp, int on_device) {
    int rc = need_adj(ctx, "rk_objective");
    if (rc) return rc;
    if (objective != RK_OBJ_HEAT && objective != RK_OBJ_DRAG) return fail(ctx, RK_EINVAL, "rk_objective: unknown objective");
    AdjState& A = *ctx->adj;
    double Jv = 0.0, dp[6];
    if ((rc = objective_impl(ctx, A, objective, &Jv, dp))) return rc;
    if (J) *J = Jv;
    if (dJdp) std::memcpy(dJdp, dp, sizeof(dp));
    if (dJdX) return store_vec(ctx, A, A.jv, dJdX, on_device);
    return RK_OK;
}

// restarted GMRES(m), right preconditioned, classical Gram-Schmidt with one
// re-orthogonalisation; Givens rotations and the small least-squares problem on the host
extern "C" int rk_adjoint_solve(rk_ctx* ctx, int objective, int32_t max_iter, double tol, int32_t* iters_done,
                                double* rel_res, double* J, double* dJdp) {
    int rc = need_adj(ctx, "rk_adjoint_solve");
    if (rc) return rc;
    if (objective != RK_OBJ_HEAT && objective != RK_OBJ_DRAG) return fail(ctx, RK_EINVAL, "rk_adjoint_solve: unknown objective");
    if (max_iter < 0 || !(tol >= 0.0)) return fail(ctx, RK_EINVAL, "rk_adjoint_solve: bad max_iter or tol");
    AdjState& A = *ctx->adj;
    cudaStream_t s = ctx->stream;
    double Jv = 0.0, dpx[6];
    if ((rc = objective_impl(ctx, A, objective, &Jv, dpx))) return rc;
    double jn = 0.0;
    if ((rc = adj_norm(ctx, A, A.jv, &jn))) return rc;
    const bool warm = A.lam_obj == objective && A.lam_ver == ctx->state_ver;
    if (!warm) CK(cudaMemsetAsync(A.lam, 0, A.np * sizeof(double), s));
    CK(adj_pc_prepare(ctx, A));
    // rv = -(A^T lam + j)
    auto residual = [&](double* beta) -> int {
        CK(adj_apply(ctx, A, A.lam, A.rv, 0.0, 0));
        vec_axpby(ctx, A, -1.0, A.jv, -1.0, A.rv);
        return adj_norm(ctx, A, A.rv, beta);
    };
    // a cold start has lam = 0: its residual is -j, its product zero
    double beta = jn;
    if (warm) {
        if ((rc = residual(&beta))) return rc;
    } else {
        vec_axpby(ctx, A, -1.0, A.jv, 0.0, A.rv);
        CK(cudaMemsetAsync(A.pout, 0, 6 * sizeof(double), s));
    }
    const int m = A.m;
    int total = 0;
    std::vector<double> H((size_t)(m + 1) * m), cs(m), sn(m), g(m + 1), y(m);
    auto Hx = [&](int i, int j) -> double& { return H[(size_t)i * m + j]; };
    while (jn > 0.0 && beta / jn > tol && total < max_iter) {
        if (!std::isfinite(beta)) return fail(ctx, RK_EDIVERGED, "rk_adjoint_solve: non-finite residual");
        vec_axpby(ctx, A, 1.0 / beta, A.rv, 0.0, A.V);
        std::fill(g.begin(), g.end(), 0.0);
        g[0] = beta;
        int jj = 0;
        for (int j = 0; j < m && total < max_iter; ++j) {
            double* Vj = A.V + (size_t)j * A.np;
            double* w = A.V + (size_t)(j + 1) * A.np;
            CK(adj_pc(ctx, A, Vj, A.tmp));
            CK(adj_apply(ctx, A, A.tmp, w, 0.0, 0));
            // two passes of classical Gram-Schmidt
            adj_mdot(ctx, A, w, A.V, j + 1, A.hd);
            rk::k_vec_msub<<<1216, 256, 0, s>>>(w, A.V, A.np, j + 1, A.hd, A.np);
            adj_mdot(ctx, A, w, A.V, j + 1, A.hd + rk::GM_MAX);
            rk::k_vec_msub<<<1216, 256, 0, s>>>(w, A.V, A.np, j + 1, A.hd + rk::GM_MAX, A.np);
            adj_mdot(ctx, A, w, w, 1, A.hd + 2 * rk::GM_MAX);
            A.launches += 2;
            CK(cudaMemcpyAsync(A.hpin, A.hd, (2 * rk::GM_MAX + 1) * sizeof(double), cudaMemcpyDeviceToHost, s));
            CK(cudaStreamSynchronize(s));
            for (int i = 0; i <= j; ++i) Hx(i, j) = A.hpin[i] + A.hpin[rk::GM_MAX + i];
            const double hn = std::sqrt(A.hpin[2 * rk::GM_MAX]);
            Hx(j + 1, j) = hn;
            if (!std::isfinite(hn)) return fail(ctx, RK_EDIVERGED, "rk_adjoint_solve: non-finite Krylov vector");
            if (hn > 0.0) vec_axpby(ctx, A, 0.0, w, 1.0 / hn, w);
            for (int i = 0; i < j; ++i) {
                const double t = cs[i] * Hx(i, j) + sn[i] * Hx(i + 1, j);
                Hx(i + 1, j) = -sn[i] * Hx(i, j) + cs[i] * Hx(i + 1, j);
                Hx(i, j) = t;
            }
            const double r = std::hypot(Hx(j, j), Hx(j + 1, j));
            cs[j] = r > 0.0 ? Hx(j, j) / r : 1.0;
            sn[j] = r > 0.0 ? Hx(j + 1, j) / r : 0.0;
            Hx(j, j) = r;
            Hx(j + 1, j) = 0.0;
            g[j + 1] = -sn[j] * g[j];
            g[j] = cs[j] * g[j];
            ++total;
            jj = j + 1;
            if (std::fabs(g[j + 1]) <= tol * jn || hn == 0.0) break;
        }
        // y = H^-1 g (upper triangular), lam += P^-1 (V y)
        for (int i = jj - 1; i >= 0; --i) {
            double t = g[i];
            for (int k = i + 1; k < jj; ++k) t -= Hx(i, k) * y[k];
            y[i] = Hx(i, i) != 0.0 ? t / Hx(i, i) : 0.0;
        }
        CK(cudaMemcpyAsync(A.hd, y.data(), jj * sizeof(double), cudaMemcpyHostToDevice, s));
        CK(cudaMemsetAsync(A.tmp2, 0, A.np * sizeof(double), s));
        rk::k_vec_madd<<<1216, 256, 0, s>>>(A.tmp2, A.V, A.np, jj, A.hd, A.np);
        A.launches++;
        CK(adj_pc(ctx, A, A.tmp2, A.tmp));
        vec_axpby(ctx, A, 1.0, A.tmp, 1.0, A.lam);
        if ((rc = residual(&beta))) return rc;
    }
    if (!std::isfinite(beta)) return fail(ctx, RK_EDIVERGED, "rk_adjoint_solve: non-finite residual");
    A.lam_obj = objective;
    A.lam_ver = ctx->state_ver;
    // total derivative: dJ/dp|_X + lam^T dR/dp (pout: from the product of the last residual)
    CK(cudaMemcpyAsync(A.hpin, A.pout, 6 * sizeof(double), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (dJdp)
        for (int j = 0; j < 6; ++j) dJdp[j] = dpx[j] + A.hpin[j];
    if (J) *J = Jv;
    if (iters_done) *iters_done = total;
    if (rel_res) *rel_res = jn > 0.0 ? beta / jn : 0.0;
    return RK_OK;
}

extern "C" int rk_adjoint_get(rk_ctx* ctx, double* lam, int on_device) {
    int rc = need_adj(ctx, "rk_adjoint_get");
    if (rc) return rc;
    if (!lam) return fail(ctx, RK_EINVAL, "rk_adjoint_get: null pointer");
    return store_vec(ctx, *ctx->adj, ctx->adj->lam, lam, on_device);
}
