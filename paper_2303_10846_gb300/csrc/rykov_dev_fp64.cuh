// Per-velocity kernels of FP64 contexts.  GB300 issues FP64 at 1/64 of its FP32 rate (one
// warp instruction per 16 cycles and SM, whatever the number of active lanes), so these
// kernels are bound by the number of FP64 instructions per (cell, velocity): they take
// comparisons on the bits, upwind signs from an FP32 dot product where its error cannot
// change the sign, and shared subexpressions wherever the formulas have them, and spend
// memory traffic (4-10 % of HBM) freely.
#pragma once

#include <algorithm>

#include "rykov_dev.cuh"

namespace rk {

// x > 0 without an FP64 comparison (false for zeros; x not NaN)
__device__ __forceinline__ bool pos_bits(double x) { return __double_as_longlong(x) > 0; }
// running extremes on the bits: of non-negative values as signed integers (start 0; a
// negative value never wins), of non-positive ones as unsigned (start -0; a positive
// value never wins)
__device__ __forceinline__ void max_bits(long long& m, double x) {
    const long long b = __double_as_longlong(x);
    m = b > m ? b : m;
}
__device__ __forceinline__ void min_bits(unsigned long long& m, double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    m = b > m ? b : m;
}
// u.n > 0 as the rounded FP64 dot product (dot_rn) has it.  The FP32 product with rounded
// u and n is off by less than 4e-7 |u|_1 (|n| <= 1) and, among subnormal numbers, 1e-44, so
// beyond thr = 1e-6 |u|_1 + 1e-43 its sign is the sign; closer, the FP64 product decides
// (beyond the range of FP32 too: thr is infinite there).
struct VelF {
    float x, y, z, thr;
};
__device__ __forceinline__ VelF vel_f(const DevBase& c, int k) {
    const float x = c.uF[k], y = c.uF[c.Kp + k], z = c.uF[2 * c.Kp + k];
    return VelF{x, y, z, fmaf(1e-6f, fabsf(x) + fabsf(y) + fabsf(z), 1e-43f)};
}
__device__ __forceinline__ bool outflow(const VelF& u, float4 n, double ux, double uy, double uz, double nx,
                                        double ny, double nz) {
    const float un = fmaf(u.z, n.z, fmaf(u.y, n.y, u.x * n.x));
    if (fabsf(un) > u.thr) return un > 0.f;
    return pos_bits(dot_rn(ux, uy, uz, nx, ny, nz));
}
// a / b for b > 0: a times the reciprocal, except near the end of the range
__device__ __forceinline__ double quot(double a, double b) {
    if (__double2hiint(b) < 0x03e00000 || __double2hiint(b) >= 0x7fc00000) return a / b;   // b < 1e-288 or huge
    return a * inv(b);
}

// Step 2 (a) in FP64 (see k_recon): one warp per cell, one velocity per lane, MS >= the
// faces of any cell (4, 6 or 8: the face loops unroll and d2 = grad phi . (x_f - x_c) is
// kept per face, so that phi(x_f - u s) = phi + L (d2 - s grad phi . u) takes two
// operations per face and field).  About 125 FP64 instructions per (cell, velocity) on
// tetrahedra against 256 of the general kernel: 4.97 -> 2.48 ms on 37,086 cells x 304
// velocities (2.65 with divisions by the library's reciprocal); BND as there.
template <int WPB, int MS, bool BND = false>
__global__ void __launch_bounds__(WPB * 32, 8)
    k_recon_d(Dev<double> c, const int* cells, int ncells, int kc) {
    __shared__ Q4<double> s_A[WPB][MS];           // LSQ weight vector, s_ij
    __shared__ Q4<double> s_B[WPB][MS];           // x_f - x_i, -
    __shared__ Q4<double> s_C[WPB][MS];           // face normal
    __shared__ float4 s_F[WPB][MS];               // face normal in FP32
    __shared__ int4 s_I[WPB][MS];                 // neighbour, face, left side
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int t = blockIdx.x * WPB + w;
    if (t >= (BND ? ncells : c.N)) return;        // whole warp
    const int i = BND ? cells[t] : t;
    const int s0 = c.slot_off[i], ns = c.slot_off[i + 1] - s0;
    if (lane < ns) {
        const int m = s0 + lane;
        const double nx = c.slot_nT[m], ny = c.slot_nT[c.nnz + m], nz = c.slot_nT[2 * c.nnz + m];
        s_A[w][lane] = Q4<double>{c.slot_lsqT[m], c.slot_lsqT[c.nnz + m], c.slot_lsqT[2 * c.nnz + m], c.slot_sT[m]};
        s_B[w][lane] = Q4<double>{c.slot_dT[m], c.slot_dT[c.nnz + m], c.slot_dT[2 * c.nnz + m], 0.0};
        s_C[w][lane] = Q4<double>{nx, ny, nz, 0.0};
        s_F[w][lane] = make_float4((float)nx, (float)ny, (float)nz, 0.f);
        s_I[w][lane] = make_int4(c.slot_nbr[m], c.slot_face[m], c.slot_left[m], 0);
    }
    __syncwarp();
    const double eps2 = c.eps2[i];
    const int limiter = (int)c.iterp[1];
    const size_t NK = (size_t)c.N * c.Kp, FK = (size_t)c.F * c.Kp;
    const size_t oi = (size_t)i * c.Kp;
    const int kend = min(c.K, (int)(blockIdx.y + 1) * kc);
    for (int k = blockIdx.y * kc + lane; k < kend; k += 32) {
        const double p[2] = {c.phi[oi + k], c.phi[NK + oi + k]};
        const double ux = c.uT[k], uy = c.uT[c.Kp + k], uz = c.uT[2 * c.Kp + k];
        double d2[2][MS], L[2], gu[2];
        if (limiter == 2) {                       // first order: phi_c itself
            L[0] = L[1] = gu[0] = gu[1] = 0.0;
#pragma unroll
            for (int q = 0; q < MS; ++q) d2[0][q] = d2[1][q] = 0.0;
        } else {
            double g[2][3] = {{0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}};
            long long hi[2] = {0, 0};
            unsigned long long lo[2] = {0x8000000000000000ull, 0x8000000000000000ull};
#pragma unroll
            for (int q = 0; q < MS; ++q) {
                if (q >= ns) break;
                const int j = s_I[w][q].x;
                if (j < 0) continue;
                const size_t oj = (size_t)j * c.Kp + k;
                const double d[2] = {c.phi[oj] - p[0], c.phi[NK + oj] - p[1]};
                const Q4<double> A = s_A[w][q];
#pragma unroll
                for (int fd = 0; fd < 2; ++fd) {
                    g[fd][0] = fma(A.x, d[fd], g[fd][0]);
                    g[fd][1] = fma(A.y, d[fd], g[fd][1]);
                    g[fd][2] = fma(A.z, d[fd], g[fd][2]);
                    max_bits(hi[fd], d[fd]);
                    min_bits(lo[fd], d[fd]);
                }
            }
            long long hi2[2] = {0, 0};
            unsigned long long lo2[2] = {0x8000000000000000ull, 0x8000000000000000ull};
#pragma unroll
            for (int q = 0; q < MS; ++q) {
                if (q >= ns) break;
                const Q4<double> B = s_B[w][q];
#pragma unroll
                for (int fd = 0; fd < 2; ++fd) {
                    d2[fd][q] = fma(g[fd][2], B.z, fma(g[fd][1], B.y, g[fd][0] * B.x));
                    max_bits(hi2[fd], d2[fd][q]);
                    min_bits(lo2[fd], d2[fd][q]);
                }
            }
            if (limiter == 3) {                   // frozen limiter values
                L[0] = c.lstore[oi + k];
                L[1] = c.lstore[NK + oi + k];
            } else if (limiter == 1 || limiter == 4) {
                // the smaller of psi(Delta_max, max d2) and psi(Delta_min, min d2), capped
                // at 1 (k_recon: the same minimum as over all faces)
#pragma unroll
                for (int fd = 0; fd < 2; ++fd) {
                    const double ep = eps2 * p[fd] * p[fd];
                    double Lv = 1.0;
                    if (hi2[fd] > 0) {
                        const double a = __longlong_as_double(hi[fd]), b = __longlong_as_double(hi2[fd]);
                        const double aa = fma(a, a, ep), b2 = b + b;
                        const double nu = fma(a, b2, aa), de = fma(a, b, fma(b2, b, aa));
                        if (nu < de) Lv = quot(nu, de);
                    }
                    if (lo2[fd] > 0x8000000000000000ull) {
                        const double a = __longlong_as_double((long long)lo[fd]), b = __longlong_as_double((long long)lo2[fd]);
                        const double aa = fma(a, a, ep), b2 = b + b;
                        const double nu = fma(a, b2, aa), de = fma(a, b, fma(b2, b, aa));
                        if (nu < Lv * de) Lv = quot(nu, de);
                    }
                    L[fd] = Lv;
                }
                if (limiter == 4) {
                    c.lstore[oi + k] = L[0];
                    c.lstore[NK + oi + k] = L[1];
                }
            } else {
                L[0] = L[1] = 1.0;
            }
#pragma unroll
            for (int fd = 0; fd < 2; ++fd) gu[fd] = fma(g[fd][2], uz, fma(g[fd][1], uy, g[fd][0] * ux));
        }
        const VelF uf = vel_f(c, k);
#pragma unroll
        for (int q = 0; q < MS; ++q) {
            if (q >= ns) break;
            const int4 I = s_I[w][q];
            if (BND && I.x >= 0) continue;
            const Q4<double> Cn = s_C[w][q];
            // the left cell is upwind where u.n > 0, the right one elsewhere
            if (outflow(uf, s_F[w][q], ux, uy, uz, Cn.x, Cn.y, Cn.z) != (I.z != 0)) continue;
            const double s = s_A[w][q].w;
            const size_t o = (size_t)I.y * c.Kp + k;
            c.face[o] = fma(L[0], fma(-s, gu[0], d2[0][q]), p[0]);
            c.face[FK + o] = fma(L[1], fma(-s, gu[1], d2[1][q]), p[1]);
        }
    }
}

// Micro flux in FP64 (see k_micro_flux): A/V folded into the normals, five FP64
// instructions per face and velocity instead of ten (735 -> 459 us on 37,086 x 304).
template <int WPB>
__global__ void __launch_bounds__(WPB * 32) k_micro_flux_d(Dev<double> c, int kc) {
    __shared__ Q4<double> s_N[WPB][MAXF];         // (A/V) n outward
    __shared__ int s_face[WPB][MAXF];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int i = blockIdx.x * WPB + w;
    if (i >= c.N) return;
    const int s0 = c.slot_off[i], ns = c.slot_off[i + 1] - s0;
    if (lane < ns) {
        const int m = s0 + lane;
        const double a = c.slot_left[m] ? c.slot_AVT[m] : -c.slot_AVT[m];
        s_N[w][lane] = Q4<double>{a * c.slot_nT[m], a * c.slot_nT[c.nnz + m], a * c.slot_nT[2 * c.nnz + m], 0.0};
        s_face[w][lane] = c.slot_face[m];
    }
    __syncwarp();
    const size_t NK = (size_t)c.N * c.Kp, FK = (size_t)c.F * c.Kp, oi = (size_t)i * c.Kp;
    const int kend = min(c.K, (int)(blockIdx.y + 1) * kc);
    for (int k = blockIdx.y * kc + lane; k < kend; k += 32) {
        const double ux = c.uT[k], uy = c.uT[c.Kp + k], uz = c.uT[2 * c.Kp + k];
        double Fg = 0.0, Fh = 0.0;
#pragma unroll 2
        for (int q = 0; q < ns; ++q) {
            const Q4<double> n = s_N[w][q];
            const size_t of = (size_t)s_face[w][q] * c.Kp + k;
            const double un = fma(uz, n.z, fma(uy, n.y, ux * n.x));
            Fg = fma(un, c.face[of], Fg);
            Fh = fma(un, c.face[FK + of], Fh);
        }
        c.res[oi + k] = Fg;
        c.res[NK + oi + k] = Fh;
    }
}

// Steps 5 and 6 in FP64 (see k_micro_sweep): the point updates of one colour, one warp
// per cell, one velocity per lane.  The first sweep stores 1/D beside Res, so that the
// later ones evaluate u.n at the inflow faces alone (D needs the outflow ones and a
// division): 16 FP64 instructions per (cell, velocity) in a middle sweep against 56.
// A launch on a quarter of 37,086 cells x 304: first 631 -> 441 us, middle 273 -> 146 us,
// last 901 -> 541 us (the first and last also with the table exponential).
// WC warps share a cell (its velocities in turn; the sums over the warps in order).
template <int WPB, int WC, bool FIRST, bool LAST>
__global__ void __launch_bounds__(WPB * 32, LAST ? 4 : 6)
    k_micro_sweep_d(Dev<double> c, const int* cells, int ncells, int colour) {
    using R = Red<double>;
    __shared__ double s_e[WPB][EQN + 2];
    __shared__ Q4<double> s_N[WPB][MAXF];         // (A/V) n outward
    __shared__ Q4<double> s_C[WPB][MAXF];         // n outward
    __shared__ float4 s_F[WPB][MAXF];             // n outward in FP32
    __shared__ int2 s_NO[WPB][MAXF];              // neighbour, neighbour term used
    __shared__ double s_S[WC > 1 && LAST ? WPB : 1][12];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    static_assert(WC == 1 || WC == WPB, "a block has whole cells: all its warps share one, or none does");
    const int t = blockIdx.x * (WPB / WC) + w / WC;
    if (t >= ncells) return;                      // whole warp (WC > 1: whole block)
    const int i = cells[t];
    const int s0 = c.slot_off[i], ns = c.slot_off[i + 1] - s0;
    if (lane < EQN + 2) s_e[w][lane] = c.ceq[(size_t)i * CEQ + lane];
    if (lane < ns) {
        const int m = s0 + lane;
        const double sg = c.slot_left[m] ? 1.0 : -1.0, a = c.slot_AVT[m];
        const double nx = sg * c.slot_nT[m], ny = sg * c.slot_nT[c.nnz + m], nz = sg * c.slot_nT[2 * c.nnz + m];
        s_N[w][lane] = Q4<double>{a * nx, a * ny, a * nz, 0.0};
        s_C[w][lane] = Q4<double>{nx, ny, nz, 0.0};
        s_F[w][lane] = make_float4((float)nx, (float)ny, (float)nz, 0.f);
        s_NO[w][lane] = make_int2(c.slot_nbr[m], (c.slot_nbr[m] >= 0) && !(FIRST && c.slot_ncol[m] > colour));
    }
    __syncwarp();
    const double* e = s_e[w];
    const double itau = e[EQN - 1], base = e[EQN];
    const size_t NK = (size_t)c.N * c.Kp, oi = (size_t)i * c.Kp;
    double a[12];
#pragma unroll
    for (int j = 0; j < 12; ++j) a[j] = 0.0;
    for (int k = lane + 32 * (w % WC); k < c.K; k += 32 * WC) {
        const double ux = c.uT[k], uy = c.uT[c.Kp + k], uz = c.uT[2 * c.Kp + k];
        const VelF uf = vel_f(c, k);
        double D = base, og = 0.0, oh = 0.0;
#pragma unroll 1
        for (int q = 0; q < ns; ++q) {
            const Q4<double> C = s_C[w][q], n = s_N[w][q];
            const int2 NO = s_NO[w][q];
            if (outflow(uf, s_F[w][q], ux, uy, uz, C.x, C.y, C.z)) {
                if (FIRST) D = fma(uz, n.z, fma(uy, n.y, fma(ux, n.x, D)));
            } else if (NO.y) {
                const size_t oj = (size_t)NO.x * c.Kp + k;
                const double dg = c.dphi[oj], dh = c.dphi[NK + oj];
                const double un = fma(uz, n.z, fma(uy, n.y, ux * n.x));
                og = fma(un, dg, og);
                oh = fma(un, dh, oh);
            }
        }
        // F in the first sweep (k_micro_flux_d), Res in the later ones
        double rg = c.res[oi + k], rh = c.res[NK + oi + k], pg = 0.0, ph = 0.0, G = 0.0, H = 0.0, iD;
        if (FIRST || LAST) {
            pg = c.phi[oi + k];
            ph = c.phi[NK + oi + k];
            eval_eq(e, ux, uy, uz, G, H);
        }
        if (FIRST) {
            rg = fma(G - pg, itau, -rg);
            rh = fma(H - ph, itau, -rh);
            c.res[oi + k] = rg;
            c.res[NK + oi + k] = rh;
            iD = inv(D);
            c.iD[oi + k] = iD;
        } else {
            iD = c.iD[oi + k];
        }
        const double xg = (rg - og) * iD, xh = (rh - oh) * iD;
        c.dphi[oi + k] = xg;
        c.dphi[NK + oi + k] = xh;
        if (LAST) {
            const double wv = c.wT[k], g1 = pg + xg, h1 = ph + xh;
            const double cx = ux - e[0], cy = uy - e[1], cz = uz - e[2];
            const double wg = wv * (g1 - G), wh = wv * (h1 - H);
            const double wc = wg * fma(cz, cz, fma(cy, cy, cx * cx));
            a[0] += wg;
            a[1] = fma(wg, ux, a[1]); a[2] = fma(wg, uy, a[2]); a[3] = fma(wg, uz, a[3]);
            a[4] = fma(c.u2h[k], wg, a[4]) + wh;
            a[5] += wh;
            a[6] = fma(wc, cx, a[6]); a[7] = fma(wc, cy, a[7]); a[8] = fma(wc, cz, a[8]);
            a[9] = fma(wh, cx, a[9]); a[10] = fma(wh, cy, a[10]); a[11] = fma(wh, cz, a[11]);
            c.phi[oi + k] = g1;
            c.phi[NK + oi + k] = h1;
        }
    }
    if (LAST) {
        warp_red0<double, 12>(a);
        if constexpr (WC > 1) {
            if (lane == 0)
#pragma unroll
                for (int j = 0; j < 12; ++j) s_S[w][j] = a[j];
            __syncthreads();
            if (threadIdx.x < 12) {
                double x = s_S[0][threadIdx.x];
                for (int q = 1; q < WC; ++q) x += s_S[q][threadIdx.x];
                c.S[(size_t)i * 12 + threadIdx.x] = x;
            }
        } else if (lane == 0) {
#pragma unroll
            for (int j = 0; j < 12; ++j) c.S[(size_t)i * 12 + j] = a[j];
        }
    }
}

// Step 2 (b)-(d) at interior faces in FP64 (see k_face_interior), as three kernels: the
// moments (one warp per face), the interface state (one thread per face) and the face
// distribution with the macro flux (one warp per face).  The state takes some 250 FP64
// instructions, powers and divisions; on one lane of a face's warp they cost what 250
// instructions of all its lanes cost (26 per velocity at K = 304), one per thread they
// vanish, for a second read of the face rows that FP64 contexts have bandwidth for.
// 71,000 faces x 304: 6.40 -> 4.09 ms (1.39 + 0.13 + 2.57; the table exponential included).
template <int WPB>
__global__ void __launch_bounds__(WPB * 32) k_face_mom_d(Dev<double> c) {
    const int lane = threadIdx.x & 31;
    const int fi = blockIdx.x * WPB + (threadIdx.x >> 5);
    if (fi >= c.Fi) return;                      // whole warp
    const int f = c.face_int[fi];
    const double* g0 = c.face + (size_t)f * c.Kp;
    const double* h0 = g0 + (size_t)c.F * c.Kp;
    float Uf[3];
    face_ref_velocity<true>(c, f, lane, Uf);
    const double Ur[3] = {(double)Uf[0], (double)Uf[1], (double)Uf[2]};
    double m[17];
#pragma unroll
    for (int j = 0; j < 17; ++j) m[j] = 0.0;
#pragma unroll 2
    for (int k = lane; k < c.K; k += 32) {
        const double w = c.wT[k], wg = w * g0[k], wh = w * h0[k];
        const double cx = c.uT[k] - Ur[0], cy = c.uT[c.Kp + k] - Ur[1], cz = c.uT[2 * c.Kp + k] - Ur[2];
        const double x = wg * cx, y = wg * cy, z = wg * cz;
        const double c2 = fma(cz, cz, fma(cy, cy, cx * cx));
        m[0] += wg; m[1] += x; m[2] += y; m[3] += z; m[4] += wh;
        m[5] = fma(x, cx, m[5]); m[6] = fma(y, cy, m[6]); m[7] = fma(z, cz, m[7]);
        m[8] = fma(x, cy, m[8]); m[9] = fma(x, cz, m[9]); m[10] = fma(y, cz, m[10]);
        m[11] = fma(x, c2, m[11]); m[12] = fma(y, c2, m[12]); m[13] = fma(z, c2, m[13]);
        m[14] = fma(wh, cx, m[14]); m[15] = fma(wh, cy, m[15]); m[16] = fma(wh, cz, m[16]);
    }
    warp_red0<double, 17>(m);
    if (lane == 0) {
        double* o = c.fmom + (size_t)fi * FMOM;
#pragma unroll
        for (int j = 0; j < 17; ++j) o[j] = m[j];
        o[17] = Ur[0]; o[18] = Ur[1]; o[19] = Ur[2];
    }
}

// feq: [0] tau/(tau + s), [1..20] make_eq's constants with s/(tau + s) folded into the
// two Maxwellians
static __global__ void __launch_bounds__(64) k_face_state_d(Dev<double> c) {
    const int fi = blockIdx.x * blockDim.x + threadIdx.x;
    if (fi >= c.Fi) return;
    const int f = c.face_int[fi];
    const double* x = c.fmom + (size_t)fi * FMOM;
    const double* Ur = x + 17;
    double e[EQN], a, b;
    face_state<double>(c, f, x, Ur, e, a, b);
    e[9] *= b;
    e[13] *= b;
    double* o = c.feq + (size_t)fi * FEQ;
    o[0] = a;
    for (int j = 0; j < 20; ++j) o[1 + j] = e[j];
}

template <int WPB>
__global__ void __launch_bounds__(WPB * 32, 8) k_face_flux_d(Dev<double> c) {
    const int lane = threadIdx.x & 31;
    const int fi = blockIdx.x * WPB + (threadIdx.x >> 5);
    if (fi >= c.Fi) return;                      // whole warp
    const int f = c.face_int[fi];
    double* g0 = c.face + (size_t)f * c.Kp;
    double* h0 = g0 + (size_t)c.F * c.Kp;
    double e[20];
    const double a = c.feq[(size_t)fi * FEQ];
#pragma unroll
    for (int j = 0; j < 20; ++j) e[j] = c.feq[(size_t)fi * FEQ + 1 + j];
    const double nx = c.fnT[f], ny = c.fnT[c.F + f], nz = c.fnT[2 * c.F + f];
    double m[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) m[j] = 0.0;
    for (int k = lane; k < c.K; k += 32) {
        const double ux = c.uT[k], uy = c.uT[c.Kp + k], uz = c.uT[2 * c.Kp + k];
        double G, H;
        eval_eq(e, ux, uy, uz, G, H);
        const double gf = fma(a, g0[k], G), hf = fma(a, h0[k], H);
        g0[k] = gf;
        h0[k] = hf;
        const double wu = c.wT[k] * fma(uz, nz, fma(uy, ny, ux * nx));
        const double wg = wu * gf;
        m[0] += wg;
        m[1] = fma(wg, ux, m[1]); m[2] = fma(wg, uy, m[2]); m[3] = fma(wg, uz, m[3]);
        m[4] = fma(wu, fma(c.u2h[k], gf, hf), m[4]);
        m[5] = fma(wu, hf, m[5]);
    }
    warp_red0<double, 6>(m);
    if (lane == 0)
#pragma unroll
        for (int d = 0; d < 6; ++d) c.mface[(size_t)f * 6 + d] = m[d];
}

// Warps per block of the FP64 kernels (the sweeps: four, below): two, so that the blocks of a small mesh spread
// evenly (an SM's FP64 pipe is the resource: 1,344 faces in blocks of eight warps left some
// SMs with twice the work of others).  Where there are fewer than FP64_FEW cells (16 warps
// per SM) the velocities of a cell are split as well, over blocks or, in the sweeps, over
// four warps.  Cavity 8^3 x 512, blocks of eight warps and no split / this rule: recon
// 178 / 84 us, faces 233 / 162, first sweeps 206 / 62, last 250 / 74.
constexpr int FP64_WPB = 2;
constexpr int FP64_FEW = 152 * 16;
static inline int vel_split_d(int K, int cells) {
    const int ns = cells >= FP64_FEW ? 1 : std::max(1, std::min((FP64_FEW + cells - 1) / cells, K / 64));
    return ((K + ns - 1) / ns + 31) / 32 * 32;
}
static inline void launch_flux_d(const Dev<double>& d, cudaStream_t s) {
    const int kc = vel_split_d(d.K, d.N);
    const dim3 g((d.N + FP64_WPB - 1) / FP64_WPB, (d.K + kc - 1) / kc);
    k_micro_flux_d<FP64_WPB><<<g, FP64_WPB * 32, 0, s>>>(d, kc);
}
template <bool FIRST, bool LAST>
static inline void launch_sweep_d(const Dev<double>& d, cudaStream_t s, const int* cells, int n, int colour) {
    if (n < FP64_FEW && d.K >= 128) k_micro_sweep_d<4, 4, FIRST, LAST><<<n, 128, 0, s>>>(d, cells, n, colour);
    else k_micro_sweep_d<4, 1, FIRST, LAST><<<(n + 3) / 4, 128, 0, s>>>(d, cells, n, colour);
}

static inline void launch_faces_d(const Dev<double>& d, cudaStream_t s) {
    constexpr int WPB = FP64_WPB;
    const int g = (d.Fi + WPB - 1) / WPB;
    k_face_mom_d<WPB><<<g, WPB * 32, 0, s>>>(d);
    k_face_state_d<<<(d.Fi + 63) / 64, 64, 0, s>>>(d);
    k_face_flux_d<WPB><<<g, WPB * 32, 0, s>>>(d);
}

// Step 1: the equilibrium distributions from the cells' constants, zero in the K padding
template <int WPB>
__global__ void __launch_bounds__(WPB * 32) k_set_eq_d(Dev<double> c) {
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * WPB + (threadIdx.x >> 5);
    if (i >= c.N) return;                         // whole warp
    double e[20];
#pragma unroll
    for (int j = 0; j < 20; ++j) e[j] = c.ceq[(size_t)i * CEQ + j];
    double* g = c.phi + (size_t)i * c.Kp;
    double* h = g + (size_t)c.N * c.Kp;
    for (int k = lane; k < c.Kp; k += 32) {
        double G = 0.0, H = 0.0;
        if (k < c.K) eval_eq(e, c.uT[k], c.uT[c.Kp + k], c.uT[2 * c.Kp + k], G, H);
        g[k] = G;
        h[k] = H;
    }
}

// the instantiation for a mesh whose cells have at most ms faces
template <bool BND>
static inline void launch_recon_d(const Dev<double>& d, cudaStream_t s, const int* cells, int n) {
    constexpr int W = FP64_WPB;
    const int kc = vel_split_d(d.K, n);
    const dim3 g((n + W - 1) / W, (d.K + kc - 1) / kc);
    if (d.ms <= 4) k_recon_d<W, 4, BND><<<g, W * 32, 0, s>>>(d, cells, n, kc);
    else if (d.ms <= 6) k_recon_d<W, 6, BND><<<g, W * 32, 0, s>>>(d, cells, n, kc);
    else k_recon_d<W, 8, BND><<<g, W * 32, 0, s>>>(d, cells, n, kc);
}

}  // namespace rk
