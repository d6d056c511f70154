// Definitions of the launch sequences (included by kern_f64.cu / kern_f32.cu only).
#pragma once

#include "rykov_dev_fp64.cuh"
#include "rykov_dev_packed.cuh"
#include "rykov_launch.cuh"

namespace rk {

constexpr int FACE_BS = 128;         // threads per boundary face
constexpr int FACE_WPB = 8;         // faces (warps) per block of the interior-face kernel
constexpr int MICRO_WPB = 8;        // cells (warps) per block of the micro sweep
constexpr int RECON_WPB = 8;        // cells (warps) per block of the reconstruction

static inline int cdiv(long long a, long long b) { return (int)((a + b - 1) / b); }

// Velocities per block (a multiple of 128) of the kernels that need no sum over them:
// kmax at most, so that the row segments in flight stay in L2, and fewer (256 at least)
// until the launch has two waves of blocks, so that a small mesh fills the GPU and its
// last wave is not nearly empty.  Middle sweep of 26,928 x 1,517: 86 -> 71 us a phase,
// recon and sweeps of the 12^3 cavity x 343: 23 -> 20, 11 -> 9 us.
static inline int vel_block(int K, long long blocks, int resident, int kmax) {
    const long long want = (2LL * resident + blocks - 1) / blocks;
    const long long ns = std::max<long long>(cdiv(K, kmax), std::min<long long>(want, cdiv(K, 256)));
    return cdiv(cdiv(K, ns), 128) * 128;
}

template <typename T>
cudaError_t Launch<T>::setup(const Dev<T>& d, cudaStream_t s) {
    k_setup_dt<T><<<d.N, 128, 0, s>>>(d);
    k_setup_lsq<T><<<cdiv(d.N, 128), 128, 0, s>>>(d);
    k_setup_face<T><<<cdiv(d.F, 256), 256, 0, s>>>(d);
    k_setup_slotT<T><<<cdiv(d.nnz > d.F ? d.nnz : d.F, 256), 256, 0, s>>>(d);
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::set_state(const Dev<T>& d, cudaStream_t s, const double* prim,
                                 const double* q) {
    k_set_state<T><<<cdiv(d.N, 64), 64, 0, s>>>(d, prim, q);
    if constexpr (std::is_same<T, double>::value)
        k_set_eq_d<FP64_WPB><<<cdiv(d.N, FP64_WPB), FP64_WPB * 32, 0, s>>>(d);
    else
        k_set_eq_p<MICRO_WPB><<<cdiv(d.N, MICRO_WPB), MICRO_WPB * 32, 0, s>>>(d);
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::begin(const Dev<T>& d, cudaStream_t s, Prof& pf) {
    k_iter_begin<T><<<1, 1, 0, s>>>(d);
    pf.launches += 1;
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::recon(const Dev<T>& d, cudaStream_t s, Prof& pf) {
    pf.begin(0, s);
    if constexpr (std::is_same<T, float>::value) {
        if (d.packed) {
            // all velocities in one block on large meshes (blocks of 512 to 2,048 velocities
            // measured 9.2 to 8.4 ms against 8.3 on 131,772 x 5,991)
            const int nb = cdiv(d.N, RECON_WPB), kc = vel_block(d.K, nb, 152 * RECONP_MINB, d.K);
            const dim3 g(nb, cdiv(d.K, kc));
            if (d.ms <= 4) {
                constexpr int sm = recon_smem(RECON_WPB);
                cudaError_t e = cudaFuncSetAttribute(k_recon_p<RECON_WPB, true>,
                                                     cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
                if (e != cudaSuccess) return e;
                k_recon_p<RECON_WPB, true><<<g, RECON_WPB * 32, sm, s>>>(d, nullptr, 0, kc);
            }
            else k_recon_p<RECON_WPB, false><<<g, RECON_WPB * 32, 0, s>>>(d, nullptr, 0, kc);
        } else
            k_recon<T, RECON_WPB><<<cdiv(d.N, RECON_WPB), RECON_WPB * 32, 0, s>>>(d);
    } else {
        launch_recon_d<false>(d, s, nullptr, d.N);
    }
    pf.end(s);
    pf.launches += 1;
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::faces_interior(const Dev<T>& d, cudaStream_t s, Prof& pf) {
    if (d.Fi) {
        pf.begin(1, s);
        if constexpr (std::is_same<T, double>::value) {
            launch_faces_d(d, s);
            pf.launches += 2;
        } else if (d.packed) {
            if (d.K > FACE_K1) k_face_interior_p<FACE_WPB, 2><<<cdiv(d.Fi, FACE_WPB / 2), FACE_WPB * 32, 0, s>>>(d);
            else k_face_interior_p<FACE_WPB, 1><<<cdiv(d.Fi, FACE_WPB), FACE_WPB * 32, 0, s>>>(d);
        } else {
            k_face_interior<T, FACE_WPB><<<cdiv(d.Fi, FACE_WPB), FACE_WPB * 32, 0, s>>>(d);
        }
        pf.end(s);
        pf.launches += 1;
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::faces_boundary(const Dev<T>& d, cudaStream_t s, Prof& pf) {
    if (d.Fb) {
        pf.begin(2, s);
        k_face_boundary<T, FACE_BS><<<d.Fb, FACE_BS, 0, s>>>(d, nullptr);
        pf.end(s);
        pf.launches += 1;
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::faces(const Dev<T>& d, cudaStream_t s, Prof& pf) {
    cudaError_t e = faces_interior(d, s, pf);
    return e != cudaSuccess ? e : faces_boundary(d, s, pf);
}

template <typename T>
cudaError_t Launch<T>::walls(const Dev<T>& d, cudaStream_t s, const int* wall_b, int nw, const int* cells,
                             int ncells, Prof& pf) {
    if (!nw) return cudaSuccess;
    k_iter_begin<T><<<1, 1, 0, s>>>(d);
    pf.begin(0, s);
    // few cells (a wall is a surface): four warps per block spread them over more SMs
    constexpr int W = 4;
    if constexpr (std::is_same<T, float>::value) {
        const dim3 g(cdiv(ncells, W), cdiv(d.K, 1024));
        if (d.packed && d.ms <= 4) k_recon_p<W, true, true><<<g, W * 32, recon_smem(W), s>>>(d, cells, ncells, 1024);
        else if (d.packed) k_recon_p<W, false, true><<<g, W * 32, 0, s>>>(d, cells, ncells, 1024);
        else k_recon<T, W, true><<<cdiv(ncells, W), W * 32, 0, s>>>(d, cells, ncells);
    } else {
        launch_recon_d<true>(d, s, cells, ncells);
    }
    pf.end(s);
    pf.begin(2, s);
    k_face_boundary<T, FACE_BS><<<nw, FACE_BS, 0, s>>>(d, wall_b);
    pf.end(s);
    pf.launches += 3;
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::radius(const Dev<T>& d, cudaStream_t s, Prof& pf) {
    pf.begin(3, s);
    k_face_radius<T><<<cdiv(d.F, 64), 64, 0, s>>>(d);
    pf.end(s);
    pf.launches += 1;
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::fluxes(const Dev<T>& d, cudaStream_t s, Prof& pf) {
    pf.begin(3, s);
    k_cell_macro_flux<T><<<cdiv(d.N, 32), 192, 0, s>>>(d);
    pf.end(s);
    pf.launches += 1;
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::micro_flux(const Dev<T>& d, cudaStream_t s, Prof& pf) {
    pf.begin(3, s);
    if constexpr (std::is_same<T, double>::value)
        launch_flux_d(d, s);
    else if (d.packed) {
        const int nb = cdiv(d.N, MICRO_WPB), kc = vel_block(d.K, nb, 152 * 3, 2048);
        k_micro_flux_p<MICRO_WPB><<<dim3(nb, cdiv(d.K, kc)), MICRO_WPB * 32, 0, s>>>(d, kc);
    } else
        k_micro_flux<T, MICRO_WPB><<<cdiv(d.N, MICRO_WPB), MICRO_WPB * 32, 0, s>>>(d);
    pf.end(s);
    pf.launches += 1;
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::macro_rec(const Dev<T>& d, cudaStream_t s, const Sched& sc, Prof& pf) {
    if (sc.macro32) return cudaSuccess;          // the FP32 form sets up in one kernel (macro)
    pf.begin(4, s);
    k_macro_rec<T><<<cdiv(d.N, 64), 64, 0, s>>>(d, sc.col_cell);
    pf.end(s);
    pf.launches += 1;
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::macro(const Dev<T>& d, cudaStream_t s, const Sched& sc, int n_macro,
                             Prof& pf) {
    pf.begin(4, s);
    const int C = (int)sc.col_off.size() - 1;
    const DevBase& db = d;
    bool first = true;               // the first phase reads what the set-up kernels wrote
    if (sc.macro32) {
        // FP32 delta form (mixed contexts)
        k_macro_prep32<T><<<cdiv(d.N, 128), 128, 0, s>>>(d);
        pf.launches += 1;
        for (const Phase& ph : sgs_phases(sc, n_macro)) {
            const int lo = sc.col_off[ph.col], n = sc.col_off[ph.col + 1] - lo, ln = sc.macro_lanes;
            const cudaError_t e = launch_phase(ln == 1 ? k_macro_sweep32<1> : ln == 4 ? k_macro_sweep32<4> : k_macro_sweep32<2>,
                                               (long long)n * ln, sc.pdl && !first, s, db, lo, n, ph.reps);
            if (e != cudaSuccess) return e;
            first = false;
            pf.launches += 1;
        }
        k_macro_finish<T><<<cdiv(d.N, 64), 64, 0, s>>>(d, 1);
        pf.end(s);
        pf.launches += 1;
        return cudaGetLastError();
    }
    k_macro_con<T><<<cdiv(d.N, 64), 64, 0, s>>>(d, sc.col_cell);
    pf.launches += 1;
    bool done = false;
    if (sc.coop_grid > 0 && n_macro > 0) {
        // all sweeps in one cooperative launch (grid barriers between colours)
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(sc.coop_grid);
        cfg.blockDim = dim3(128);
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cudaError_t e = cudaLaunchKernelEx(&cfg, k_macro_coop<T>, d, d.col_off_d, C, n_macro, d.bar,
                                           sc.coop_extra, sc.coop_limit_ns);
        if (e == cudaSuccess) {
            pf.launches += 1;
            done = true;
        } else {
            (void)cudaGetLastError();
        }
    }
    if (!done) {
        for (const Phase& ph : sgs_phases(sc, n_macro)) {
            const int lo = sc.col_off[ph.col], n = sc.col_off[ph.col + 1] - lo, L = macro_lanes(n, d.ms);
            const cudaError_t e = launch_phase(L == 1 ? k_macro_sweep<1, MACRO_INC<T>> : L == 2 ? k_macro_sweep<2, MACRO_INC<T>>
                                               : L == 4 ? k_macro_sweep<4, MACRO_INC<T>> : k_macro_sweep<8, MACRO_INC<T>>,
                                               (long long)n * L, sc.pdl && !first, s, db, lo, n, ph.reps);
            if (e != cudaSuccess) return e;
            first = false;
            pf.launches += 1;
        }
    }
    k_macro_finish<T><<<cdiv(d.N, 64), 64, 0, s>>>(d, 0);
    pf.end(s);
    pf.launches += 1;
    return cudaGetLastError();
}

// dynamic shared memory of one block of the staged micro sweep
template <typename T>
struct StBytes {
    template <bool FIRST, bool LAST>
    static size_t get(int maxs) {
        return (size_t)MICRO_ST_WPB * 2 * (2 * maxs + 4) * 32 * micro_nv<T, FIRST, LAST>() * sizeof(T);
    }
};

template <typename T>
cudaError_t Launch<T>::micro(const Dev<T>& d, cudaStream_t s, const Sched& sc, int n_micro,
                             Prof& pf) {
    const int nsw = 2 * n_micro;
    // A phase that repeats the colour of the one before changes nothing (the increment of
    // a cell depends on its neighbours only, and they are of other colours), so the three
    // repeats at the turns are dropped: 13 of 16 phases are left with four colours and two
    // iterations, 5 of 8 with two.  The update of the last
    // sweep then joins the phase before it.  The one repeat that stays is the first
    // sweep's directly before the last sweep's (n_micro = 1), which form Res and the
    // update in different kernels.
    std::vector<Phase> phases;
    for (const Phase& ph : sgs_phases(sc, n_micro)) {
        const int last = ph.sweep + ph.reps - 1;                    // sweep of its last repeat
        if (ph.sweep == 0 && ph.reps > 1 && last == nsw - 1) {
            phases.push_back(Phase{ph.col, 0, 1});
            phases.push_back(Phase{ph.col, nsw - 1, 1});
        } else {
            phases.push_back(Phase{ph.col, last == nsw - 1 ? last : ph.sweep, 1});
        }
    }
    for (const Phase& ph : phases) {
        const int sw = ph.sweep, col = ph.col;
        const int lo = sc.col_off[col], n = sc.col_off[col + 1] - lo;
        // the first sweep forms Res for every cell of this colour; the last
        // sweep applies the update and the Step-6 sums
        pf.begin(sw == 0 ? 5 : (sw == nsw - 1 ? 7 : 6), s);
        const int* cl = sc.col_cell + lo;
        const int kind = sw == 0 ? 0 : (sw == nsw - 1 ? 2 : 1);
        if constexpr (std::is_same<T, double>::value) {
            if (sw == 0) launch_sweep_d<true, false>(d, s, cl, n, col);
            else if (sw == nsw - 1) launch_sweep_d<false, true>(d, s, cl, n, col);
            else launch_sweep_d<false, false>(d, s, cl, n, col);
        } else {
            if (d.packed && ((sc.staged >> kind) & 1)) {
                constexpr int W = MICRO_ST_WPB;
                const dim3 g(cdiv(n, W)), b(W * 32);
                const int mx = sc.maxs;
                const size_t sb = sw == 0 ? StBytes<T>::template get<true, false>(mx)
                                          : (sw == nsw - 1 ? StBytes<T>::template get<false, true>(mx)
                                                           : StBytes<T>::template get<false, false>(mx));
                if ((sc.staged >> 3) & 1) {            // the cell's own rows by bulk copies
                    if (sw == 0) k_micro_sweep_st_p<W, true, false, true><<<g, b, sb, s>>>(d, cl, n, col, mx);
                    else if (sw == nsw - 1) k_micro_sweep_st_p<W, false, true, true><<<g, b, sb, s>>>(d, cl, n, col, mx);
                    else k_micro_sweep_st_p<W, false, false, true><<<g, b, sb, s>>>(d, cl, n, col, mx);
                } else {
                    if (sw == 0) k_micro_sweep_st_p<W, true, false, false><<<g, b, sb, s>>>(d, cl, n, col, mx);
                    else if (sw == nsw - 1) k_micro_sweep_st_p<W, false, true, false><<<g, b, sb, s>>>(d, cl, n, col, mx);
                    else k_micro_sweep_st_p<W, false, false, false><<<g, b, sb, s>>>(d, cl, n, col, mx);
                }
            } else if (d.packed) {
                const int nb = cdiv(n, MICRO_WPB);
                const int kc = vel_block(d.K, nb, 152 * (sw == 0 ? MICROP_FIRST_MINB : MICROP_MID_MINB), 2048);
                const dim3 g(nb, sw == nsw - 1 ? 1 : cdiv(d.K, kc)), b(MICRO_WPB * 32);
                if (sw == 0) k_micro_sweep_p<MICRO_WPB, true, false><<<g, b, 0, s>>>(d, cl, n, col, kc);
                else if (sw == nsw - 1) k_micro_sweep_p<MICRO_WPB, false, true><<<g, b, 0, s>>>(d, cl, n, col, 0);
                else k_micro_sweep_p<MICRO_WPB, false, false><<<g, b, 0, s>>>(d, cl, n, col, kc);
            } else if ((sc.staged >> kind) & 1) {
                constexpr int W = MICRO_ST_WPB;
                const dim3 g(cdiv(n, W)), b(W * 32);
                const int mx = sc.maxs;
                if (sw == 0)
                    k_micro_sweep_st<T, W, true, false><<<g, b, StBytes<T>::template get<true, false>(mx), s>>>(d, cl, n, col, mx);
                else if (sw == nsw - 1)
                    k_micro_sweep_st<T, W, false, true><<<g, b, StBytes<T>::template get<false, true>(mx), s>>>(d, cl, n, col, mx);
                else
                    k_micro_sweep_st<T, W, false, false><<<g, b, StBytes<T>::template get<false, false>(mx), s>>>(d, cl, n, col, mx);
            } else {
                const dim3 g(cdiv(n, MICRO_WPB)), b(MICRO_WPB * 32);
                if (sw == 0) k_micro_sweep<T, MICRO_WPB, true, false><<<g, b, 0, s>>>(d, cl, n, col);
                else if (sw == nsw - 1) k_micro_sweep<T, MICRO_WPB, false, true><<<g, b, 0, s>>>(d, cl, n, col);
                else k_micro_sweep<T, MICRO_WPB, false, false><<<g, b, 0, s>>>(d, cl, n, col);
            }
        }
        pf.end(s);
        pf.launches += 1;
    }
    pf.begin(8, s);
    k_cell_update<T><<<cdiv(d.N, 128), 128, 0, s>>>(d);
    k_residual_reduce<T><<<1, 384, 0, s>>>(d, cdiv(d.N, 128));
    pf.end(s);
    pf.launches += 2;
    return cudaGetLastError();
}

template <typename T>
size_t Launch<T>::micro_staged_smem(int maxs) {
    // FP64 sweeps wait for the FP64 pipe, not for loads: no staged form
    if constexpr (std::is_same<T, double>::value) {
        (void)maxs;
        return 0;
    } else {
    const size_t need = StBytes<T>::template get<true, false>(maxs) > StBytes<T>::template get<false, true>(maxs)
                            ? StBytes<T>::template get<true, false>(maxs) : StBytes<T>::template get<false, true>(maxs);
    const size_t need2 = need > StBytes<T>::template get<false, false>(maxs) ? need : StBytes<T>::template get<false, false>(maxs);
    int dev = 0, lim = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&lim, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return 0;
    // the kernels' static shared memory comes on top of the dynamic part
    if (need2 + 4096 > (size_t)lim) return 0;
    constexpr int W = MICRO_ST_WPB;
    if (cudaFuncSetAttribute(k_micro_sweep_st<T, W, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)StBytes<T>::template get<true, false>(maxs)) != cudaSuccess ||
        cudaFuncSetAttribute(k_micro_sweep_st<T, W, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)StBytes<T>::template get<false, true>(maxs)) != cudaSuccess ||
        cudaFuncSetAttribute(k_micro_sweep_st<T, W, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)StBytes<T>::template get<false, false>(maxs)) != cudaSuccess)
        return 0;
    {
        const int b0 = (int)StBytes<T>::template get<true, false>(maxs);
        const int b1 = (int)StBytes<T>::template get<false, true>(maxs);
        const int b2 = (int)StBytes<T>::template get<false, false>(maxs);
        constexpr auto A = cudaFuncAttributeMaxDynamicSharedMemorySize;
        if (cudaFuncSetAttribute(k_micro_sweep_st_p<W, true, false, false>, A, b0) != cudaSuccess ||
            cudaFuncSetAttribute(k_micro_sweep_st_p<W, false, true, false>, A, b1) != cudaSuccess ||
            cudaFuncSetAttribute(k_micro_sweep_st_p<W, false, false, false>, A, b2) != cudaSuccess ||
            cudaFuncSetAttribute(k_micro_sweep_st_p<W, true, false, true>, A, b0) != cudaSuccess ||
            cudaFuncSetAttribute(k_micro_sweep_st_p<W, false, true, true>, A, b1) != cudaSuccess ||
            cudaFuncSetAttribute(k_micro_sweep_st_p<W, false, false, true>, A, b2) != cudaSuccess)
            return 0;
    }
    return need2;
    }
}

template <typename T>
cudaError_t Launch<T>::debug_micro_flux(const Dev<T>& d, cudaStream_t s, T* out) {
    dim3 grid(d.N, cdiv(d.K, 128));
    k_debug_micro_flux<T><<<grid, 128, 0, s>>>(d, out);
    return cudaGetLastError();
}

template <typename T>
int Launch<T>::coop_blocks_per_sm() {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_macro_coop<T>, 128, 0) != cudaSuccess) return 0;
    return n;
}

template <typename T>
cudaError_t Launch<T>::temps(const Dev<T>& d, cudaStream_t s, double* out) {
    k_temps<T><<<cdiv(d.N, 256), 256, 0, s>>>(d, out);
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::surface(const Dev<T>& d, cudaStream_t s, const int* wall_b, int nw,
                               double p_inf, double qdyn, double Umag, double* out,
                               double* contrib, double* tot) {
    if (nw) k_surface<T><<<cdiv(nw, 128), 128, 0, s>>>(d, wall_b, nw, p_inf, qdyn, Umag, out, contrib);
    k_sum4<<<1, 256, 0, s>>>(contrib, nw, tot);
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::aero(const Dev<T>& d, cudaStream_t s, const int* wall_b, int nw,
                            const double x_ref[3], double* contrib, double* tot) {
    if (nw) k_aero<T><<<cdiv(nw, 128), 128, 0, s>>>(d, wall_b, nw, x_ref[0], x_ref[1], x_ref[2], contrib);
    k_sum6<<<1, 256, 0, s>>>(contrib, nw, tot);
    return cudaGetLastError();
}

}  // namespace rk
