// Launch sequences of librykov, one explicit instantiation per precision
// (kern_f64.cu: double, kern_f32.cu: float).  Every function enqueues on `s` and
// returns cudaSuccess or the first launch error.
#pragma once

#include <algorithm>
#include <vector>

#include "rykov_dev.cuh"

namespace rk {

// Launch accounting and optional per-class CUDA-event timing (rk_profile).
struct Prof {
    bool on = false;
    long long launches = 0;
    std::vector<cudaEvent_t> ev;      // pool, created on enable
    std::vector<int> cls;             // class of each recorded pair
    size_t used = 0;                  // events used (2 per pair)
    void begin(int c, cudaStream_t s) {
        if (!on) return;
        if (used + 2 > ev.size()) {
            size_t n = ev.size();
            ev.resize(n ? 2 * n : 1024);
            for (size_t i = n; i < ev.size(); ++i) cudaEventCreate(&ev[i]);
        }
        cudaEventRecord(ev[used], s);
        cls.push_back(c);
    }
    void end(cudaStream_t s) {
        if (!on) return;
        cudaEventRecord(ev[used + 1], s);
        used += 2;
    }
};

struct Sched {
    const int* col_cell;            // device: cells grouped by colour
    std::vector<int> col_off;       // host: colour offsets (C+1)
    int coop_grid = 0;              // blocks of the cooperative macro solve (0: per-colour launches)
    unsigned coop_extra = 0;        // test only: barrier arrivals that never come
    unsigned long long coop_limit_ns = 1000000000ull;   // bound of every barrier wait
    int maxs = 0;                   // most faces of one cell
    int staged = 0;                 // micro sweeps with staged (asynchronous) row loads:
                                    // bit 0 first sweep, bit 1 middle sweeps, bit 2 last;
                                    // bit 3: the cell's own rows by bulk copies (packed)
    int macro32 = 0;                // macro PR-SGS in FP32 delta form (mixed contexts)
    int pdl = 0;                    // macro colour phases launched with programmatic
                                    // stream serialisation
    int macro_lanes = 4;            // threads per cell of the FP32 macro phases (1, 2, 4)
};

// The colour phases of n PR-SGS iterations (each a forward and a backward sweep over the
// colours that have cells), with consecutive phases of one colour counted as repeats of
// the first: at every turn the next sweep begins with the colour that the last one
// ended with, whose cells see unchanged neighbours.  Of the 16 phases of two micro
// iterations with four colours 13 are left, of the 320 of 40 macro iterations 241 (with
// two colours 5 of 8 and 81 of 160), with the same bits.  Measured per iteration, before
// and after: cavity 12^3 x 343 (mixed) 1.375 -> 0.805 ms, sphere 61,911 x 3,033 (mixed)
// 13.71 -> 12.29 ms, sphere 37,086 x 304 (FP64) 23.6 -> 22.3 ms; the adjoint's
// preconditioner takes the same list: GMRES(10) on 5,911 x 304 176 -> 155 ms.
struct Phase {
    int col, sweep, reps;
};
static inline std::vector<Phase> sgs_phases(const Sched& sc, int n) {
    const int C = (int)sc.col_off.size() - 1;
    std::vector<Phase> ph;
    for (int sw = 0; sw < 2 * n; ++sw)
        for (int cc = 0; cc < C; ++cc) {
            const int col = (sw & 1) ? C - 1 - cc : cc;
            if (sc.col_off[col + 1] == sc.col_off[col]) continue;
            if (!ph.empty() && ph.back().col == col) ph.back().reps++;
            else ph.push_back(Phase{col, sw, 1});
        }
    return ph;
}

// Whether the macro phases of a context are launched ahead of their turn (programmatic
// stream serialisation), unless RYKOV_PDL says otherwise: always in mixed contexts
// (iteration with / without: cavity 12^3 x 343 0.41 / 0.45 ms, sphere 26,928 x 1,517 with the
// FP32 solve 2.77 / 2.92, cone 75,177 x 7,980 28.4 / 28.8); in FP64 contexts only while the
// largest phase leaves SMs free (cavity 8^3 x 512 0.65 / 0.71), since waiting blocks hold up
// the FP64 micro flux beside them (sphere 37,086 x 304 13.6 / 13.2)
static inline bool macro_ahead(const std::vector<int>& col_off, int ms, bool fp64) {
    int n = 0;
    for (size_t c = 0; c + 1 < col_off.size(); ++c) n = std::max(n, col_off[c + 1] - col_off[c]);
    return !fp64 || (long long)n * macro_lanes(n, ms) < 152LL * MACRO_BS;
}

// one colour phase, with programmatic stream serialisation if pdl
template <typename... A, typename... B>
static inline cudaError_t launch_phase(void (*k)(A...), long long threads, bool pdl, cudaStream_t s, const B&... args) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((threads + MACRO_BS - 1) / MACRO_BS));
    cfg.blockDim = dim3(MACRO_BS);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, static_cast<A>(args)...);
}

template <typename T>
struct Launch {
    static cudaError_t setup(const Dev<T>& d, cudaStream_t s);
    static cudaError_t set_state(const Dev<T>& d, cudaStream_t s, const double* prim,
                                 const double* q);
    static cudaError_t begin(const Dev<T>& d, cudaStream_t s, Prof& pf);   // schedule of the iteration
    static cudaError_t recon(const Dev<T>& d, cudaStream_t s, Prof& pf);
    static cudaError_t faces(const Dev<T>& d, cudaStream_t s, Prof& pf);   // interior + boundary
    static cudaError_t faces_interior(const Dev<T>& d, cudaStream_t s, Prof& pf);
    static cudaError_t faces_boundary(const Dev<T>& d, cudaStream_t s, Prof& pf);
    // the boundary faces of a list (indices into face_bnd) and the reconstruction at the
    // boundary faces of the listed cells: the faces that the wall quantities need
    static cudaError_t walls(const Dev<T>& d, cudaStream_t s, const int* wall_b, int nw, const int* cells,
                             int ncells, Prof& pf);
    static cudaError_t radius(const Dev<T>& d, cudaStream_t s, Prof& pf);  // spectral radii of W^n
    static cudaError_t fluxes(const Dev<T>& d, cudaStream_t s, Prof& pf);
    // micro flux F into res: independent of the macro solve (a parallel graph branch)
    static cudaError_t micro_flux(const Dev<T>& d, cudaStream_t s, Prof& pf);
    // set-up of the macro solve that needs W^n and the radii only; macro does the rest
    static cudaError_t macro_rec(const Dev<T>& d, cudaStream_t s, const Sched& sc, Prof& pf);
    static cudaError_t macro(const Dev<T>& d, cudaStream_t s, const Sched& sc, int n_macro,
                             Prof& pf);
    static cudaError_t micro(const Dev<T>& d, cudaStream_t s, const Sched& sc, int n_micro,
                             Prof& pf);
    // shared memory of the staged micro sweeps for a mesh with at most maxs faces per
    // cell (0 if it exceeds the device limit); sets the kernels' attribute
    static size_t micro_staged_smem(int maxs);
    static cudaError_t debug_micro_flux(const Dev<T>& d, cudaStream_t s, T* out);
    static cudaError_t temps(const Dev<T>& d, cudaStream_t s, double* out);
    static int coop_blocks_per_sm();
    static cudaError_t surface(const Dev<T>& d, cudaStream_t s, const int* wall_b, int nw,
                               double p_inf, double qdyn, double Umag, double* out,
                               double* contrib, double* tot);
    static cudaError_t aero(const Dev<T>& d, cudaStream_t s, const int* wall_b, int nw,
                            const double x_ref[3], double* contrib, double* tot);
};

extern template struct Launch<double>;
extern template struct Launch<float>;

}  // namespace rk
