// Device side of the adjoint of the steady residual operator (FP64, or FP32 per-velocity
// arithmetic for mixed-precision contexts).
//
// Unknowns X = (phi, W, q) of a steady state of the implicit iteration (Sec. 3.5 with
// dphi = 0 and a zero macro increment), residual R(X; p) = (R_phi, R_W, R_q):
//   R_phi = (phi*(W, q) - phi)/tau(W) - F(phi; p)          Eq. implicit_mic_final_equ
//   R_W   = sum_k w Psi (phi - phi*)  (+ rho R((1-1/Z) T_rot + T/Z) - rho E_rot in
//           the rotational-energy row)                      Eqs. solve_rho - solve_Erot
//   R_q   = 1/2 sum_k w c|c|^2 (g - g*) + (a_tr - 1) q_tr,
//           sum_k w c (h - h*) + (a_rot - 1) q_rot           Eqs. solve_qtr, solve_qrot
// F is the micro flux of Eq. implicit_mic_flux with the interface distribution of
// Eq. flux_solve_phi and the limited reconstruction of Eq. flux_solve_phi_phi.
// Parameters p = (T_w shift of every wall, rho_inf, U_inf[3], T_inf of every farfield).
//
// The kernels below apply (dR/dX)^T v and (dR/dp)^T v by hand-written reverse mode of
// the forward kernels: per cell (collision terms and the compensation rows), per
// interior face (moments -> interface state -> phi* -> blend), per boundary face
// (wall density rho_w, farfield Maxwellian), and the gradient / Venkatakrishnan
// limiter / least-squares gather.  Every scatter of the forward pass becomes a gather
// in a fixed order, so results are bit-reproducible.
#pragma once

#include "rykov_dev_fp64.cuh"

namespace rk {

constexpr int ADJ_FPAR = 12;     // per boundary face: dR/dp^T v (6), J, force (3), 2 spare
// records of the state (written once per state): equilibrium constants of a cell or an
// interior face (EQA), the face's moments (FMOM, as the forward kernels'), and the sums
// over the velocities that depend on v
constexpr int EQA = 22, ADJ_NS = 15, ADJ_CS = 20, ADJ_FS = 17, ADJ_FC = 16;

// Arrays in the arithmetic type S of the per-velocity work: FP64, or FP32 for mixed
// contexts, whose vectors, scalars and sums stay FP64
template <typename S>
struct AdjArr {
    const S *u, *w;              // [3][Kp], [Kp]
    const S *phi, *v;            // [2][N][Kp] the state, the phi block of v
    const S *f0;                 // [2][F][Kp] phi(x_f - u s)
    S *fbar;                     // [2][F][Kp] its adjoint
    S *oc;                       // [2][N][Kp] the cell terms of the output
    S *nb;                       // [2][ms][N][Kp] what a cell's gradient and limiter give its neighbours
    S *iD;                       // [N][Kp] inverse diagonal of the transposed micro sweeps
    const S* lstore;             // [2][N][Kp] frozen limiter values
    S *ceq, *feq, *fcoef;        // [N][EQA], [Fi][EQA], [Fi][ADJ_FC]
};
struct AdjBufs {
    double* ophi;                // [2][N][Kp] output (phi part)
    const double *vW, *vq;       // [N][6]
    double *oW, *oq;             // [N][6]
    const int* slot_mirg;        // [nnz] global slot of the same face in the neighbour's list (-1)
    const double* slot_AVn;      // [nnz] A_f / V_neighbour (0 at boundary faces)
    const double* tau;           // [N] tau(W_i)
    double *fmom, *fsum, *csum;  // [Fi][FMOM], [Fi][ADJ_FS + 1], [N][ADJ_CS]
    double* fpar;                // [Fb][ADJ_FPAR]
    const double* iterp;         // [4]: [1] reconstruction mode of the steady operator (0-3)
    double obj_scale;            // weight of the objective seed at wall faces (0: none)
    int objective;               // 0: heat to the wall, 1: drag
    double edrag[3];             // drag direction
};

// velocities per lane and step, and their loads
template <typename S>
__host__ __device__ constexpr int adj_nv() { return sizeof(S) == 4 ? 4 : 1; }
// Sums over the velocities: FP64 sums; in FP32 the terms of a step's four velocities are
// added plainly, the steps with compensation (with every term compensated the product on
// 61,911 x 1,517 took 11.30 instead of 11.04 ms, and the W rows' error of 2.3e-7 changed by
// 2 %: it is that of the terms)
template <typename S, int N>
struct AdjSum {
    Acc<S> a[N];
    S t[N];
    __device__ __forceinline__ void begin() {
        if constexpr (sizeof(S) == 4)
#pragma unroll
            for (int j = 0; j < N; ++j) t[j] = S(0);
    }
    __device__ __forceinline__ S* terms() {
        if constexpr (sizeof(S) == 4) return t;
        else return &a[0].s;
    }
    __device__ __forceinline__ void end() {
        if constexpr (sizeof(S) == 4)
#pragma unroll
            for (int j = 0; j < N; ++j) a[j].add(t[j]);
    }
    // totals over the warp, written by lane 0 (FP32: as float-float pairs; Red<S>::load turns
    // them into FP64 in the thread-per-cell and thread-per-face kernels, where the
    // conversions do not cost a whole warp's FP64 slots each)
    __device__ __forceinline__ void store(double* out, int lane) {
        typename Red<S>::V v[N];
#pragma unroll
        for (int j = 0; j < N; ++j) v[j] = Red<S>::from(a[j]);
        warp_red0<S, N>(v);
        if (lane == 0)
#pragma unroll
            for (int j = 0; j < N; ++j) Red<S>::store(out + j, v[j]);
    }
};
template <typename S, int N>
__device__ __forceinline__ void adj_sums(const double* p, double (&t)[N]) {
#pragma unroll
    for (int j = 0; j < N; ++j) t[j] = Red<S>::load(p + j);
}
static_assert(sizeof(Acc<double>) == sizeof(double), "running FP64 sums are an array of doubles");

// ------------------------------------------------------------------------------------
// reverse mode of one Rykov equilibrium point (Eqs. eqdf_G* - eqdf_Rrot)
// ------------------------------------------------------------------------------------
// State in the variables of the formula: theta = R T, theta_tr = R T_tr,
// theta_rot = R T_rot.  With p = rho theta etc., s = c.q_tr, r = c.q_rot and the weights
// 1 - 1/Z and 1/Z in the Maxwellians M_t (at theta_tr) and M (at theta),
//   G* = M_t (1 + s A_t) + M (1 + s A),  A_t = (|c|^2/theta_tr - 5) / (15 rho theta_tr^2),
//                                        A = w0 (|c|^2/theta - 5) / (15 rho theta^2)
//   R* = theta_rot M_t (1 + s A_t) + B_t r M_t + theta M (1 + s A) + B r M,
//        B_t = (1 - delta) / (rho theta_tr),  B = w1 (1 - delta) / (rho theta).
// For weights (Gb, Hb) of (G*, R*) the derivatives with respect to the state are sums over
// the velocities of a few products, with P = (Gb + theta_rot Hb) M_t, Q = Hb M_t,
// P' = (Gb + theta Hb) M, Q' = Hb M, E = P (1 + s A_t) + B_t r Q, E' likewise,
// v1 = B_t Q + B Q', v2 = P A_t + P' A, y = |c|^2/theta, k' = w0/(15 rho theta^2), y_t and k alike:
//   rho          (1/rho) sum (P + P')          (the heat-flux terms cancel)
//   theta_rot    sum Q (1 + s A_t)
//   theta        (1/theta) sum theta Q' (1 + s A) - B r Q' + k' s P' (10 - 3 y) + E' (y - 3)/2;
//                theta_tr likewise without the first
//   q_rot, q_tr  sum v1 c, sum v2 c
//   U            sum ((E - 2 k s P)/theta_tr + (E' - 2 k' s P')/theta) c - q_rot sum v1 - q_tr sum v2
// Fifteen sums and about 95 operations a velocity, against 190 for the chain rule written
// out term by term.  Sums: 0 rho, 1 theta_rot, 2 theta, 3 theta_tr (2 and 3 without the
// factors 1/theta), 4 v1, 5 v2, 6-8 v1 c, 9-11 v2 c, 12-14 the U sum.  No constant has more
// than 1/(rho theta^2) in it, so that FP32 serves any units that the forward form does
// (with 1/(rho theta^4), theta = 7e10 lost the derivatives of the temperatures).
// Constants (EqA, EQA values in memory): see eqa_make.
template <typename S>
struct EqA {
    S U[3], qt[3], qr[3], thr, th, nt, n, ka, kb, kc, kd, Bt, B, itr, it, ib;
};
static_assert(sizeof(EqA<double>) == EQA * sizeof(double), "EQA");
// scale: factor on the Maxwellians (the blend's weight b at a face; ib = 1/b)
template <typename S, typename T>
__device__ __forceinline__ EqA<S> eqa_make(const Dev<T>& c, double rho, const double* U, double T_, double Ttr,
                                           double Trot, const double* qtr, const double* qrot, double scale) {
    const double th = c.R * T_, tt = c.R * Ttr, it = 1.0 / th, itr = 1.0 / tt, ir = 1.0 / rho;
    const double i15 = ir / 15.0;
    EqA<S> e;
    for (int k = 0; k < 3; ++k) { e.U[k] = (S)U[k]; e.qt[k] = (S)qtr[k]; e.qr[k] = (S)qrot[k]; }
    e.thr = (S)(c.R * Trot);
    e.th = (S)th;
    const double at = 2.0 * PI * tt, ar = 2.0 * PI * th;
    e.nt = (S)(scale * (1.0 - 1.0 / c.Z) * rho / (at * sqrt(at)));
    e.n = (S)(scale / c.Z * rho / (ar * sqrt(ar)));
    const double ka = itr * itr * i15, kc = c.omega0 * it * it * i15;
    e.ka = (S)ka; e.kb = (S)(-5.0 * ka);
    e.kc = (S)kc; e.kd = (S)(-5.0 * kc);
    e.Bt = (S)((1.0 - c.delta) * ir * itr);
    e.B = (S)(c.omega1 * (1.0 - c.delta) * ir * it);
    e.itr = (S)itr; e.it = (S)it;
    e.ib = (S)(1.0 / scale);
    return e;
}
// adds the 15 products at velocity u to t; G, H receive G*, R* (times the scale)
template <typename S>
__device__ __forceinline__ void eqa_terms(const EqA<S>& e, S ux, S uy, S uz, S Gb, S Hb, S* t, S& G, S& H) {
    const S cx = ux - e.U[0], cy = uy - e.U[1], cz = uz - e.U[2];
    const S c2 = cx * cx + cy * cy + cz * cz;
    const S s = cx * e.qt[0] + cy * e.qt[1] + cz * e.qt[2];
    const S r = cx * e.qr[0] + cy * e.qr[1] + cz * e.qr[2];
    const S yt = c2 * e.itr, y = c2 * e.it, hl = S(-0.5 * 1.4426950408889634);
    const S Mt = e.nt * ex2(yt * hl), M = e.n * ex2(y * hl);
    const S At = yt * e.ka + e.kb, A = y * e.kc + e.kd;
    const S sAt = s * At, sA = s * A;
    const S Gt = Mt * sAt + Mt, Gr = M * sA + M;
    const S BM = e.Bt * Mt + e.B * M;
    G = Gt + Gr;
    H = e.thr * Gt + (e.th * Gr + r * BM);
    const S P = (Hb * e.thr + Gb) * Mt, Q = Hb * Mt, P1 = (Hb * e.th + Gb) * M, Q1 = Hb * M;
    const S Qr = Q * r * e.Bt, Q1r = Q1 * r * e.B, kP = P * s * e.ka, kP1 = P1 * s * e.kc;
    const S E = P * sAt + (P + Qr), E1 = P1 * sA + (P1 + Q1r), tQ = e.th * Q1;
    t[0] += P + P1;
    t[1] += Q * sAt + Q;
    t[2] += tQ * sA + tQ;
    t[2] += kP1 * (S(10) - S(3) * y);
    t[2] += E1 * (S(0.5) * y - S(1.5));
    t[2] -= Q1r;
    t[3] += kP * (S(10) - S(3) * yt);
    t[3] += E * (S(0.5) * yt - S(1.5));
    t[3] -= Qr;
    const S v1 = Hb * BM, v2 = P * At + P1 * A;
    t[4] += v1;
    t[5] += v2;
    t[6] += v1 * cx; t[7] += v1 * cy; t[8] += v1 * cz;
    t[9] += v2 * cx; t[10] += v2 * cy; t[11] += v2 * cz;
    const S g = e.itr * (E - S(2) * kP) + e.it * (E1 - S(2) * kP1);
    t[12] += g * cx; t[13] += g * cy; t[14] += g * cz;
}
// derivatives with respect to (rho, U, theta, theta_tr, theta_rot, q_tr, q_rot) from the
// fifteen sums (d in the order of the comment above eqa_terms' formulas: 0 rho, 1-3 U,
// 4 theta, 5 theta_tr, 6 theta_rot, 7-9 q_tr, 10-12 q_rot)
__device__ __forceinline__ void eqa_grad(const double* t, double rho, double th, double tt, const double* qtr,
                                         const double* qrot, double (&d)[13]) {
    d[0] = t[0] / rho;
    for (int k = 0; k < 3; ++k) {
        d[1 + k] = t[12 + k] - qrot[k] * t[4] - qtr[k] * t[5];
        d[7 + k] = t[9 + k];
        d[10 + k] = t[6 + k];
    }
    d[4] = t[2] / th;
    d[5] = t[3] / tt;
    d[6] = t[1];
}

// ------------------------------------------------------------------------------------
// cell terms: collision part of R_phi and the compensation rows R_W, R_q
// ------------------------------------------------------------------------------------
// per state: tau(W_i) and the constants of phi*(W_i, q_i), one thread per cell
template <typename S>
__global__ void __launch_bounds__(64) k_adj_cstate(Dev<double> c, double* tau, S* ceq) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= c.N) return;
    const Prim p = prim_from_W(c.W + 6 * (size_t)i, c.R);
    const double* q = c.q + 6 * (size_t)i;
    const double t = relax_time(c, p.rho, p.Ttr);
    tau[i] = t;
    EqA<S> e = eqa_make<S>(c, p.rho, p.U, p.T, p.Ttr, p.Trot, q, q + 3, 1.0);
    e.ib = (S)(1.0 / t);                 // a cell's record: 1/tau in the place of 1/scale
    *reinterpret_cast<EqA<S>*>(ceq + (size_t)i * EQA) = e;
}

// One warp per cell.  OUT: write the cell part of (dR/dphi)^T v (the gathers add the flux
// part); the compensation rows' weights (vW, vq) enter unless ZERO says that they are zero.
// The sums for oW, oq (k_adj_crev): 0-14 the equilibrium's, 15 sum v.(phi* - phi),
// 16 sum w dg |c|^2, 17-19 sum w dg (c.vq_tr) c; and sum w dh times vq_rot in 12-14
// (the U sum: both are derivatives through c = u - U with the opposite sign of eqa's).
template <int WPB, typename S, bool OUT, bool ZERO>
__global__ void __launch_bounds__(WPB * 32) k_adj_cell(Dev<double> c, AdjBufs a, AdjArr<S> r) {
    constexpr int NV = adj_nv<S>();
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * WPB + (threadIdx.x >> 5);
    if (i >= c.N) return;
    const EqA<S> st = *reinterpret_cast<const EqA<S>*>(r.ceq + (size_t)i * EQA);
    const S it = st.ib;
    S vW[6], vq[6], vl = S(0);
    if (!ZERO && lane < 12) vl = (S)(lane < 6 ? a.vW[6 * (size_t)i + lane] : a.vq[6 * (size_t)i + lane - 6]);
#pragma unroll
    for (int d = 0; d < 6; ++d) {
        vW[d] = ZERO ? S(0) : __shfl_sync(0xffffffffu, vl, d);
        vq[d] = ZERO ? S(0) : __shfl_sync(0xffffffffu, vl, 6 + d);
    }
    const size_t NK = (size_t)c.N * c.Kp, oi = (size_t)i * c.Kp;
    AdjSum<S, ADJ_CS> m;
    for (int k0 = NV * lane; k0 < c.K; k0 += 32 * NV) {
        S ux[NV], uy[NV], uz[NV], w[NV], g[NV], h[NV], vg[NV], vh[NV], og[NV], oh[NV];
        vload(r.u + k0, ux);
        vload(r.u + c.Kp + k0, uy);
        vload(r.u + 2 * c.Kp + k0, uz);
        vload(r.w + k0, w);
        vload(r.phi + oi + k0, g);
        vload(r.phi + NK + oi + k0, h);
        vload(r.v + oi + k0, vg);
        vload(r.v + NK + oi + k0, vh);
        m.begin();
        S* t = m.terms();
#pragma unroll
        for (int e = 0; e < NV; ++e) {
            S Gb = vg[e] * it, Hb = vh[e] * it, G, H;
            const S cx = ux[e] - st.U[0], cy = uy[e] - st.U[1], cz = uz[e] - st.U[2];
            const S c2 = cx * cx + cy * cy + cz * cz;
            S cvt = S(0);
            if (!ZERO) {
                // weights of phi in the compensation rows (moments Psi and the heat fluxes)
                cvt = cx * vq[0] + cy * vq[1] + cz * vq[2];
                const S cvr = cx * vq[3] + cy * vq[4] + cz * vq[5] + (vW[4] + vW[5]);
                const S u2h = S(0.5) * (ux[e] * ux[e] + uy[e] * uy[e] + uz[e] * uz[e]);
                const S mg = ux[e] * vW[1] + uy[e] * vW[2] + uz[e] * vW[3] + (u2h * vW[4] + vW[0]) + S(0.5) * c2 * cvt;
                Gb -= w[e] * mg;
                Hb -= w[e] * cvr;
            }
            og[e] = -Gb;
            oh[e] = -Hb;
            if (k0 + e < c.K) {              // (the K padding: no equilibrium terms)
                eqa_terms(st, ux[e], uy[e], uz[e], Gb, Hb, t, G, H);
                const S dg = g[e] - G, dh = h[e] - H;
                t[15] -= vg[e] * dg;
                t[15] -= vh[e] * dh;
                if (!ZERO) {
                    const S wd = w[e] * dg, x = wd * cvt, wh = w[e] * dh;
                    t[16] += wd * c2;
                    t[17] += x * cx; t[18] += x * cy; t[19] += x * cz;
                    t[12] -= wh * vq[3]; t[13] -= wh * vq[4]; t[14] -= wh * vq[5];
                }
            } else {
                og[e] = oh[e] = S(0);
            }
        }
        m.end();
        if (OUT) {
            vstore(r.oc + oi + k0, og);
            vstore(r.oc + NK + oi + k0, oh);
        }
    }
    m.store(a.csum + (size_t)i * ADJ_CS, lane);
}

// oW, oq from the sums: the reverse of the primitives, tau and the scalar parts of the
// compensation rows.  One thread per cell.
template <typename S>
__global__ void __launch_bounds__(64) k_adj_crev(Dev<double> c, AdjBufs a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= c.N) return;
    const double R = c.R, Z = c.Z;
    const double* q = c.q + 6 * (size_t)i;
    const Prim p = prim_from_W(c.W + 6 * (size_t)i, R);
    const double tau = a.tau[i], itau = 1.0 / tau;
    double t[ADJ_CS];
    adj_sums<S>(a.csum + (size_t)i * ADJ_CS, t);
    const double *vW = a.vW + 6 * (size_t)i, *vq = a.vq + 6 * (size_t)i;
    double d[13];
    eqa_grad(t, p.rho, R * p.T, R * p.Ttr, q, q + 3, d);
    double rb = d[0], Ub[3];
    for (int k = 0; k < 3; ++k) Ub[k] = d[1 + k] - 0.5 * vq[k] * t[16] - t[17 + k];
    double Tb = R * d[4], Ttrb = R * d[5], Trotb = R * d[6];
    const double taub = -t[15] * itau * itau;
    double qb[6];
    for (int k = 0; k < 6; ++k) qb[k] = d[7 + k];
    double Wb[6] = {0.0, 0.0, 0.0, 0.0, 0.0, -vW[5]};
    // rotational-energy row: + rho R ((1 - 1/Z) T_rot + T/Z) - rho E_rot
    rb += vW[5] * R * ((1.0 - 1.0 / Z) * p.Trot + p.T / Z);
    Trotb += vW[5] * p.rho * R * (1.0 - 1.0 / Z);
    Tb += vW[5] * p.rho * R / Z;
    // heat-flux rows: + (a - 1) q
    const double atr = (1.0 / 3.0) * (1.0 - (1.0 - c.omega0) / Z);
    const double arot = (1.0 - c.delta) * (1.0 - (1.0 - c.omega1) / Z);
    for (int k = 0; k < 3; ++k) { qb[k] += vq[k] * (atr - 1.0); qb[3 + k] += vq[3 + k] * (arot - 1.0); }
    // tau = mu(T_tr) / (rho R T_tr); d ln mu / d ln T_tr from the viscosity law
    Ttrb += taub * tau * (viscosity_slope(c, p.Ttr) - 1.0) / p.Ttr;
    rb -= taub * tau / p.rho;
    // primitives from W
    const double k15 = 1.0 / (1.5 * p.rho * R), k25 = 1.0 / (2.5 * p.rho * R), kr = 1.0 / (p.rho * R);
    double keb = 0.0;
    Wb[4] += Ttrb * k15; keb -= Ttrb * k15; Wb[5] -= Ttrb * k15; rb -= Ttrb * p.Ttr / p.rho;
    Wb[5] += Trotb * kr; rb -= Trotb * p.Trot / p.rho;
    Wb[4] += Tb * k25; keb -= Tb * k25; rb -= Tb * p.T / p.rho;
    const double U2 = p.U[0] * p.U[0] + p.U[1] * p.U[1] + p.U[2] * p.U[2];
    rb += keb * 0.5 * U2;
    double UbU = 0.0;
    for (int k = 0; k < 3; ++k) {
        Ub[k] += keb * p.rho * p.U[k];
        Wb[1 + k] += Ub[k] / p.rho;
        UbU += Ub[k] * p.U[k];
    }
    rb -= UbU / p.rho;
    Wb[0] += rb;
    for (int k = 0; k < 6; ++k) { a.oW[6 * (size_t)i + k] = Wb[k]; a.oq[6 * (size_t)i + k] = qb[k]; }
}

// ------------------------------------------------------------------------------------
// steady residual R(X; p) from the face distributions phi_ij in c.face (forward face
// kernels run first): R_phi into a.ophi, R_W into a.oW, R_q into a.oq.  One warp per cell.
// ------------------------------------------------------------------------------------
template <int WPB>
__global__ void __launch_bounds__(WPB * 32) k_adj_residual(Dev<double> c, AdjBufs a) {
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * WPB + (threadIdx.x >> 5);
    if (i >= c.N) return;
    const double R = c.R, Z = c.Z;
    const double* W = c.W + 6 * (size_t)i;
    const double* q = c.q + 6 * (size_t)i;
    const Prim p = prim_from_W(W, R);
    const double itau = 1.0 / relax_time(c, p.rho, p.Ttr);
    double e[EQN];
    make_eq<double, double>(c, p.rho, p.U, p.T, p.Ttr, p.Trot, q, q + 3, e);
    const size_t NK = (size_t)c.N * c.Kp, FK = (size_t)c.F * c.Kp;
    const int s0 = c.slot_off[i], s1 = c.slot_off[i + 1];
    double S[12];
#pragma unroll
    for (int j = 0; j < 12; ++j) S[j] = 0.0;
    for (int k = lane; k < c.K; k += 32) {
        const double ux = c.u[k], uy = c.u[c.Kp + k], uz = c.u[2 * c.Kp + k], w = c.w[k];
        double Fg = 0.0, Fh = 0.0;
        for (int m = s0; m < s1; ++m) {
            const int f = c.slot_face[m];
            double un = dot_rn(ux, uy, uz, c.fn[f], c.fn[c.F + f], c.fn[2 * c.F + f]);
            if (!c.slot_left[m]) un = -un;
            Fg += c.slot_AV[m] * un * c.face[(size_t)f * c.Kp + k];
            Fh += c.slot_AV[m] * un * c.face[FK + (size_t)f * c.Kp + k];
        }
        double G, H;
        eval_eq(e, ux, uy, uz, G, H);
        const size_t o = (size_t)i * c.Kp + k;
        const double g = c.phi[o], h = c.phi[NK + o];
        a.ophi[o] = (G - g) * itau - Fg;
        a.ophi[NK + o] = (H - h) * itau - Fh;
        const double dg = g - G, dh = h - H;
        const double cx = ux - p.U[0], cy = uy - p.U[1], cz = uz - p.U[2];
        const double c2 = cx * cx + cy * cy + cz * cz;
        S[0] += w * dg;
        S[1] += w * ux * dg; S[2] += w * uy * dg; S[3] += w * uz * dg;
        S[4] += w * (0.5 * (ux * ux + uy * uy + uz * uz) * dg + dh);
        S[5] += w * dh;
        S[6] += w * cx * c2 * dg; S[7] += w * cy * c2 * dg; S[8] += w * cz * c2 * dg;
        S[9] += w * cx * dh; S[10] += w * cy * dh; S[11] += w * cz * dh;
    }
    warp_sum<12>(S);
    if (lane != 0) return;
    double* oW = a.oW + 6 * (size_t)i;
    double* oq = a.oq + 6 * (size_t)i;
    for (int d = 0; d < 5; ++d) oW[d] = S[d];
    oW[5] = S[5] + p.rho * R * ((1.0 - 1.0 / Z) * p.Trot + p.T / Z) - W[5];
    const double atr = (1.0 / 3.0) * (1.0 - (1.0 - c.omega0) / Z);
    const double arot = (1.0 - c.delta) * (1.0 - (1.0 - c.omega1) / Z);
    for (int d = 0; d < 3; ++d) {
        oq[d] = 0.5 * S[6 + d] + (atr - 1.0) * q[d];
        oq[3 + d] = S[9 + d] + (arot - 1.0) * q[3 + d];
    }
}

// ------------------------------------------------------------------------------------
// interior faces: reverse of Step 2 (b)-(d)
//   k_adj_mom     (per state) the 17 moments of phi0 = phi(x_f - u s) about U_r, the mean of
//                 the cells' velocities, as in the forward kernels
//   k_adj_fstate  (per state, one thread per face) interface state -> constants of phi*
//   k_adj_face_a  adjoint of phi_ij, wb = -A (u.n)(v_L/V_L - v_R/V_R): the sums of phi*'s
//                 state derivatives and of the blend's tau derivative
//   k_adj_frev    (one thread per face) reverse of the interface state down to the moments
//   k_adj_face_b  adjoint of phi0, written to fbar
// The scalar chains (some 700 FP64 instructions a face) ran on every lane of the face's
// warp before; the moments and states are formed once per state, not once per product.
// One product with its state, before and after: 37,706 faces x 304 FP64 7.96 -> 4.0 ms
// (moments 0.72, sums 2.40, fbar 0.77, scalars 0.08), 125,693 x 1,517 FP32 12.6 -> 2.9 ms.
// ------------------------------------------------------------------------------------
// interface state from the moments: everything that the reverse needs
struct AdjFace {
    double rho, U[3], Er0, T, Ttr0, tau, den, Erot, Trot, Ttr, Q[6], S[6], dtr, drot, qtr[3], qrot[3];
};
template <typename S, typename T>
__device__ __forceinline__ AdjFace adj_face(const Dev<T>& c, const double* mom, double s) {
    AdjFace f;
    double x[17];
    adj_sums<S>(mom, x);
    const double Rg = c.R, Z = c.Z, ir = 1.0 / x[0];
    f.rho = x[0];
    const double d[3] = {x[1] * ir, x[2] * ir, x[3] * ir};
    for (int k = 0; k < 3; ++k) f.U[k] = mom[17 + k] + d[k];
    const double tr = x[5] + x[6] + x[7], dd = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    const double etr = 0.5 * (tr - f.rho * dd), i15 = 1.0 / (1.5 * f.rho * Rg);
    f.Er0 = x[4];
    f.T = (etr + f.Er0) / (2.5 * f.rho * Rg);
    f.Ttr0 = etr * i15;
    f.tau = relax_time(c, f.rho, f.Ttr0);
    f.den = Z * f.tau + s;
    f.Erot = (Z * f.tau * f.Er0 + s * f.rho * Rg * f.T) / f.den;
    f.Trot = f.Erot / (f.rho * Rg);
    f.Ttr = (etr + f.Er0 - f.Erot) * i15;
    // sums about U: sum w c|c|^2 g, sum w c h (Q) and sum w c c g (S: xx yy zz xy xz yz)
    const double Sd[3] = {x[5] * d[0] + x[8] * d[1] + x[9] * d[2], x[8] * d[0] + x[6] * d[1] + x[10] * d[2],
                          x[9] * d[0] + x[10] * d[1] + x[7] * d[2]};
    for (int k = 0; k < 3; ++k) {
        f.Q[k] = x[11 + k] - 2.0 * Sd[k] - tr * d[k] + 2.0 * f.rho * dd * d[k];
        f.Q[3 + k] = x[14 + k] - d[k] * f.Er0;
        f.S[k] = x[5 + k] - f.rho * d[k] * d[k];
    }
    f.S[3] = x[8] - f.rho * d[0] * d[1];
    f.S[4] = x[9] - f.rho * d[0] * d[2];
    f.S[5] = x[10] - f.rho * d[1] * d[2];
    f.dtr = f.tau + s - s / 3.0 * (1.0 - 1.0 / Z + c.omega0 / Z);
    f.drot = f.tau + s - s * (1.0 - c.delta) * (1.0 - 1.0 / Z + c.omega1 / Z);
    for (int k = 0; k < 3; ++k) {
        f.qtr[k] = f.tau * 0.5 * f.Q[k] / f.dtr;
        f.qrot[k] = f.tau * f.Q[3 + k] / f.drot;
    }
    return f;
}

template <int WPB, typename S>
__global__ void __launch_bounds__(WPB * 32) k_adj_mom(Dev<double> c, AdjBufs a, AdjArr<S> r) {
    constexpr int NV = adj_nv<S>();
    const int lane = threadIdx.x & 31;
    const int fi = blockIdx.x * WPB + (threadIdx.x >> 5);
    if (fi >= c.Fi) return;
    const int f = c.face_int[fi];
    const S* g0 = r.f0 + (size_t)f * c.Kp;
    const S* h0 = g0 + (size_t)c.F * c.Kp;
    float Ur[3];
    face_ref_velocity<sizeof(S) == 8>(c, f, lane, Ur);
    AdjSum<S, 17> m;
    for (int k0 = NV * lane; k0 < c.K; k0 += 32 * NV) {
        S ux[NV], uy[NV], uz[NV], w[NV], g[NV], h[NV];
        vload(r.u + k0, ux);
        vload(r.u + c.Kp + k0, uy);
        vload(r.u + 2 * c.Kp + k0, uz);
        vload(r.w + k0, w);
        vload(g0 + k0, g);
        vload(h0 + k0, h);
        m.begin();
        S* t = m.terms();
#pragma unroll
        for (int e = 0; e < NV; ++e) {
            const S cx = ux[e] - (S)Ur[0], cy = uy[e] - (S)Ur[1], cz = uz[e] - (S)Ur[2];
            const S wg = w[e] * g[e], wh = w[e] * h[e], x = wg * cx, y = wg * cy, z = wg * cz;
            const S c2 = cx * cx + cy * cy + cz * cz;
            t[0] += wg; t[1] += x; t[2] += y; t[3] += z; t[4] += wh;
            t[5] += x * cx; t[6] += y * cy; t[7] += z * cz; t[8] += x * cy; t[9] += x * cz; t[10] += y * cz;
            t[11] += x * c2; t[12] += y * c2; t[13] += z * c2;
            t[14] += wh * cx; t[15] += wh * cy; t[16] += wh * cz;
        }
        m.end();
    }
    double* o = a.fmom + (size_t)fi * FMOM;
    m.store(o, lane);
    if (lane == 0)
        for (int d = 0; d < 3; ++d) o[17 + d] = (double)Ur[d];
}

template <typename S>
__global__ void __launch_bounds__(64) k_adj_fstate(Dev<double> c, AdjBufs a, AdjArr<S> r) {
    const int fi = blockIdx.x * blockDim.x + threadIdx.x;
    if (fi >= c.Fi) return;
    const double s = c.fs[c.face_int[fi]];
    const AdjFace f = adj_face<S>(c, a.fmom + (size_t)fi * FMOM, s);
    *reinterpret_cast<EqA<S>*>(r.feq + (size_t)fi * EQA) =
        eqa_make<S>(c, f.rho, f.U, f.T, f.Ttr, f.Trot, f.qtr, f.qrot, s / (f.tau + s));
}

// wb = -A (u.n)(v_L/V_L - v_R/V_R) of both fields
template <typename S>
struct AdjSeed {
    S nx, ny, nz, il, ir;
    const S *vl, *vr;
    size_t NK;
    __device__ __forceinline__ AdjSeed(const Dev<double>& c, const AdjArr<S>& r, int f) {
        const double A = -c.fa[f];
        const int l = c.fc[2 * f], q = c.fc[2 * f + 1];
        nx = (S)(A * c.fn[f]); ny = (S)(A * c.fn[c.F + f]); nz = (S)(A * c.fn[2 * c.F + f]);
        il = (S)(1.0 / c.vol[l]);
        ir = (S)(1.0 / c.vol[q]);
        vl = r.v + (size_t)l * c.Kp;
        vr = r.v + (size_t)q * c.Kp;
        NK = (size_t)c.N * c.Kp;
    }
    template <int NV>
    __device__ __forceinline__ void get(int k0, const S (&ux)[NV], const S (&uy)[NV], const S (&uz)[NV], S (&wg)[NV],
                                        S (&wh)[NV]) const {
        S a[NV], b[NV], d[NV], e[NV];
        vload(vl + k0, a);
        vload(vr + k0, b);
        vload(vl + NK + k0, d);
        vload(vr + NK + k0, e);
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const S un = ux[q] * nx + uy[q] * ny + uz[q] * nz;
            wg[q] = un * (a[q] * il - b[q] * ir);
            wh[q] = un * (d[q] * il - e[q] * ir);
        }
    }
};

// sums 0-14 of the equilibrium (times b), 15 sum wb.(phi0 - phi*)
template <int WPB, typename S>
__global__ void __launch_bounds__(WPB * 32) k_adj_face_a(Dev<double> c, AdjBufs a, AdjArr<S> r) {
    constexpr int NV = adj_nv<S>();
    const int lane = threadIdx.x & 31;
    const int fi = blockIdx.x * WPB + (threadIdx.x >> 5);
    if (fi >= c.Fi) return;
    const int f = c.face_int[fi];
    const S* g0 = r.f0 + (size_t)f * c.Kp;
    const S* h0 = g0 + (size_t)c.F * c.Kp;
    const EqA<S> st = *reinterpret_cast<const EqA<S>*>(r.feq + (size_t)fi * EQA);
    const AdjSeed<S> seed(c, r, f);
    AdjSum<S, 16> m;
    for (int k0 = NV * lane; k0 < c.K; k0 += 32 * NV) {
        S ux[NV], uy[NV], uz[NV], g[NV], h[NV], wg[NV], wh[NV];
        vload(r.u + k0, ux);
        vload(r.u + c.Kp + k0, uy);
        vload(r.u + 2 * c.Kp + k0, uz);
        vload(g0 + k0, g);
        vload(h0 + k0, h);
        seed.get(k0, ux, uy, uz, wg, wh);
        m.begin();
        S* t = m.terms();
#pragma unroll
        for (int e = 0; e < NV; ++e) {
            if (k0 + e >= c.K) continue;     // (the K padding: no equilibrium terms)
            S G, H;
            eqa_terms(st, ux[e], uy[e], uz[e], wg[e], wh[e], t, G, H);
            t[15] += wg[e] * (g[e] - st.ib * G);
            t[15] += wh[e] * (h[e] - st.ib * H);
        }
        m.end();
    }
    m.store(a.fsum + (size_t)fi * (ADJ_FS + 1), lane);
}

// reverse of the interface state; coefficients of pass B:
// 0 a, 1 rho, 2-4 momentum, 5 energy, 6 energy + rotational, 7-9 Q_tr, 10-12 Q_rot, 13-15 U
template <typename S>
__global__ void __launch_bounds__(64) k_adj_frev(Dev<double> c, AdjBufs a, AdjArr<S> r) {
    const int fi = blockIdx.x * blockDim.x + threadIdx.x;
    if (fi >= c.Fi) return;
    const double Rg = c.R, Z = c.Z, s = c.fs[c.face_int[fi]];
    const AdjFace f = adj_face<S>(c, a.fmom + (size_t)fi * FMOM, s);
    double t[16];
    adj_sums<S>(a.fsum + (size_t)fi * (ADJ_FS + 1), t);
    const double rho = f.rho, tau = f.tau, ts = tau + s;
    double d[13];
    eqa_grad(t, rho, Rg * f.T, Rg * f.Ttr, f.qtr, f.qrot, d);
    double rb = d[0], Ub[3] = {d[1], d[2], d[3]};
    double Tb = Rg * d[4], Ttrb = Rg * d[5], Trotb = Rg * d[6], taub = t[15] * s / (ts * ts);
    double Qtb[3], Qrb[3];
    for (int k = 0; k < 3; ++k) {
        Qtb[k] = d[7 + k] * tau * 0.5 / f.dtr;
        taub += d[7 + k] * 0.5 * f.Q[k] * (f.dtr - tau) / (f.dtr * f.dtr);
        Qrb[k] = d[10 + k] * tau / f.drot;
        taub += d[10 + k] * f.Q[3 + k] * (f.drot - tau) / (f.drot * f.drot);
    }
    {   // heat-flux sums depend on U through c = u - U
        const double P2 = f.S[0] + f.S[1] + f.S[2];
        const double M[3][3] = {{f.S[0], f.S[3], f.S[4]}, {f.S[3], f.S[1], f.S[5]}, {f.S[4], f.S[5], f.S[2]}};
        for (int e = 0; e < 3; ++e) {
            double x = Qtb[e] * P2 + Qrb[e] * f.Er0;
            for (int k = 0; k < 3; ++k) x += 2.0 * Qtb[k] * M[k][e];
            Ub[e] -= x;
        }
    }
    const double k15 = 1.0 / (1.5 * rho * Rg), k25 = 1.0 / (2.5 * rho * Rg);
    double Eb = Ttrb * k15, keb = -Ttrb * k15, Erotb = -Ttrb * k15;
    rb -= Ttrb * f.Ttr / rho;
    Erotb += Trotb / (rho * Rg);
    rb -= Trotb * f.Trot / rho;
    taub += Erotb * Z * (f.Er0 - f.Erot) / f.den;
    double Er0b = Erotb * Z * tau / f.den;
    rb += Erotb * s * Rg * f.T / f.den;
    Tb += Erotb * s * rho * Rg / f.den;
    const double Ttr0b = taub * tau * (viscosity_slope(c, f.Ttr0) - 1.0) / f.Ttr0;
    rb -= taub * tau / rho;
    Eb += Ttr0b * k15; keb -= Ttr0b * k15; Er0b -= Ttr0b * k15;
    rb -= Ttr0b * f.Ttr0 / rho;
    Eb += Tb * k25; keb -= Tb * k25;
    rb -= Tb * f.T / rho;
    const double U2 = f.U[0] * f.U[0] + f.U[1] * f.U[1] + f.U[2] * f.U[2];
    rb += keb * 0.5 * U2;
    S* o = r.fcoef + (size_t)fi * ADJ_FC;
    double UbU = 0.0;
    for (int k = 0; k < 3; ++k) {
        Ub[k] += keb * rho * f.U[k];
        o[2 + k] = (S)(Ub[k] / rho);
        UbU += Ub[k] * f.U[k];
        o[7 + k] = (S)Qtb[k];
        o[10 + k] = (S)Qrb[k];
        o[13 + k] = (S)f.U[k];
    }
    rb -= UbU / rho;
    o[0] = (S)(tau / ts);
    o[1] = (S)rb;
    o[5] = (S)Eb;
    o[6] = (S)(Eb + Er0b);
}

template <int WPB, typename S>
__global__ void __launch_bounds__(WPB * 32) k_adj_face_b(Dev<double> c, AdjBufs a, AdjArr<S> r) {
    constexpr int NV = adj_nv<S>();
    const int lane = threadIdx.x & 31;
    const int fi = blockIdx.x * WPB + (threadIdx.x >> 5);
    if (fi >= c.Fi) return;
    const int f = c.face_int[fi];
    S q[ADJ_FC];
#pragma unroll
    for (int j = 0; j < ADJ_FC; ++j) q[j] = r.fcoef[(size_t)fi * ADJ_FC + j];
    const AdjSeed<S> seed(c, r, f);
    S* gb = r.fbar + (size_t)f * c.Kp;
    S* hb = gb + (size_t)c.F * c.Kp;
    for (int k0 = NV * lane; k0 < c.K; k0 += 32 * NV) {
        S ux[NV], uy[NV], uz[NV], w[NV], wg[NV], wh[NV];
        vload(r.u + k0, ux);
        vload(r.u + c.Kp + k0, uy);
        vload(r.u + 2 * c.Kp + k0, uz);
        vload(r.w + k0, w);
        seed.get(k0, ux, uy, uz, wg, wh);
#pragma unroll
        for (int e = 0; e < NV; ++e) {
            const S cx = ux[e] - q[13], cy = uy[e] - q[14], cz = uz[e] - q[15];
            const S c2 = cx * cx + cy * cy + cz * cz;
            const S u2h = S(0.5) * (ux[e] * ux[e] + uy[e] * uy[e] + uz[e] * uz[e]);
            const S x = q[1] + q[2] * ux[e] + q[3] * uy[e] + q[4] * uz[e] + q[5] * u2h +
                        c2 * (q[7] * cx + q[8] * cy + q[9] * cz);
            const S y = q[6] + q[10] * cx + q[11] * cy + q[12] * cz;
            wg[e] = q[0] * wg[e] + w[e] * x;
            wh[e] = q[0] * wh[e] + w[e] * y;
        }
        vstore(gb + k0, wg);
        vstore(hb + k0, wh);
    }
}

// u.n > 0 as the reconstruction of the same arithmetic decides it
template <typename S>
__device__ __forceinline__ bool adj_outflow(const VelF& u, float4 n, S ux, S uy, S uz, const Q4<S>& N) {
    if constexpr (sizeof(S) == 8) return outflow(u, n, ux, uy, uz, N.x, N.y, N.z);
    else return dot_rn(ux, uy, uz, N.x, N.y, N.z) > S(0);
}

// ------------------------------------------------------------------------------------
// boundary faces: reverse of the wall / farfield treatment (no interface collision).
// Seeds: -A (u.n) v_i / V_i from R_phi, plus obj_scale times the derivative of the
// objective at wall faces (heat: A w (u.n)(|u|^2/2 g + h); drag: A w (u.n)(u.e) g).
// Writes fbar at outgoing velocities and per face fpar = (dT_w, drho_inf, dU_inf[3],
// dT_inf, J_f, force_f[3]).  One block per boundary face, FP64 arithmetic on the FP64 vector
// (v: its phi block, rows of ldv doubles), in FP32 contexts too: (dR/dp)^T v comes from here
// alone, and fbar is rounded once, when it is stored.
// ------------------------------------------------------------------------------------
template <int BS, typename S>
__global__ void __launch_bounds__(BS) k_adj_face_boundary(Dev<double> c, AdjBufs a, AdjArr<S> r, const double* v,
                                                          int ldv) {
    constexpr int NW = BS / 32;
    __shared__ double red[NW][6], sh[8], mc[8];
    const int b = blockIdx.x;
    const int f = c.face_bnd[b];
    const int bc = -1 - c.fc[2 * f + 1];
    const int i = c.fc[2 * f];
    const bool wall = c.bck[bc] == 0;
    const size_t FK = (size_t)c.F * c.Kp;
    const S* g0 = r.f0 + (size_t)f * c.Kp;
    const S* h0 = g0 + FK;
    S* gbar = r.fbar + (size_t)f * c.Kp;
    S* hbar = gbar + FK;
    const double nx = c.fn[f], ny = c.fn[c.F + f], nz = c.fn[2 * c.F + f], A = c.fa[f];
    const float4 nf = make_float4((float)nx, (float)ny, (float)nz, 0.f);
    const double* bv = c.bcv + 5 * bc;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    // the upwind decision of the reconstruction and of the gather, on their values of u and n:
    // f0 holds, and the gather reads, the velocities that leave the cell by that decision
    auto leaves = [&](int k) {
        VelF uf{};
        if constexpr (sizeof(S) == 8) uf = vel_f(c, k);
        return adj_outflow(uf, nf, r.u[k], r.u[c.Kp + k], r.u[2 * c.Kp + k], Q4<S>{(S)nx, (S)ny, (S)nz, S(0)});
    };
    if (threadIdx.x == 0) {
        const double T = bv[4], RT = c.R * T, an = 2.0 * PI * RT;
        mc[0] = (wall ? 1.0 : bv[0]) / (an * sqrt(an));
        mc[1] = -0.5 * 1.4426950408889634 / RT;              // exponent of 2
        mc[2] = 0.5 / (RT * T);                               // dM/dT = M (|c|^2 mc2 - mc3)
        mc[3] = 1.5 / T;
        mc[4] = RT;
        mc[5] = -A / c.vol[i];
        mc[6] = 1.0 / RT;
    }
    __syncthreads();
    const double RT = mc[4], sv = mc[5], seed = wall ? a.obj_scale : 0.0;
    const double *vg = v + (size_t)i * ldv, *vh = vg + (size_t)c.N * ldv;
    // adjoint of g_ij at velocity k: -A (u.n) v / V and the objective's seed
    auto g_seed = [&](int k, double un, double wu, double u2h, double ux, double uy, double uz) {
        double x = sv * un * vg[k];
        if (seed != 0.0)
            x += seed * A * wu * (a.objective == 0 ? u2h : ux * a.edrag[0] + uy * a.edrag[1] + uz * a.edrag[2]);
        return x;
    };
    // |c|^2 and M at velocity k
    auto maxw = [&](int k, double& cx, double& cy, double& cz, double& c2) {
        cx = c.u[k] - bv[1];
        cy = c.u[c.Kp + k] - bv[2];
        cz = c.u[2 * c.Kp + k] - bv[3];
        c2 = cx * cx + cy * cy + cz * cz;
        return mc[0] * ex2(c2 * mc[1]);
    };
    auto block_total = [&](auto& acc, auto nn) {
        constexpr int N = decltype(nn)::value;
        warp_red0<double, N>(acc);
        if (lane == 0)
            for (int j = 0; j < N; ++j) red[wib][j] = acc[j];
        __syncthreads();
        if (threadIdx.x < N) {
            double t = red[0][threadIdx.x];
            for (int q = 1; q < NW; ++q) t += red[q][threadIdx.x];
            sh[threadIdx.x] = t;
        }
        __syncthreads();
    };
    double rw = 1.0, num = 0.0, dn = 0.0, dnT = 0.0;
    if (wall) {
        double v[3] = {0.0, 0.0, 0.0};       // outflow, inflow of M, its T derivative
        for (int k = threadIdx.x; k < c.K; k += BS) {
            const double ux = c.u[k], uy = c.u[c.Kp + k], uz = c.u[2 * c.Kp + k];
            const double wu = c.w[k] * (ux * nx + uy * ny + uz * nz);
            if (leaves(k)) {
                v[0] += wu * (double)g0[k];
            } else {
                double cx, cy, cz, c2;
                const double M = maxw(k, cx, cy, cz, c2);
                v[1] -= wu * M;
                v[2] -= wu * (M * (c2 * mc[2] - mc[3]));
            }
        }
        block_total(v, std::integral_constant<int, 3>());
        num = sh[0]; dn = sh[1]; dnT = sh[2];
        rw = num / dn;
        __syncthreads();
    }
    // wall: 0 rho_w adjoint, 1 T_w adjoint (direct), 2 J_f (heat), 3-5 force_f;
    // farfield: 0 rho_inf, 1-3 U_inf, 4 T_inf
    double acc[6] = {0, 0, 0, 0, 0, 0};
    for (int k = threadIdx.x; k < c.K; k += BS) {
        const double ux = c.u[k], uy = c.u[c.Kp + k], uz = c.u[2 * c.Kp + k], w = c.w[k];
        const double un = ux * nx + uy * ny + uz * nz, wu = w * un;
        const double u2h = 0.5 * (ux * ux + uy * uy + uz * uz);
        const double wgb = g_seed(k, un, wu, u2h, ux, uy, uz);
        double whb = sv * un * vh[k];
        if (seed != 0.0 && a.objective == 0) whb += seed * A * wu;
        double gf = 0.0, hf = 0.0;
        if (leaves(k)) {
            if (seed != 0.0) {               // J and the force: of the objective only
                gf = (double)g0[k];
                hf = (double)h0[k];
            }
            if (!wall) gbar[k] = (S)wgb;     // (walls: below, with the share through rho_w)
            hbar[k] = (S)whb;
        } else {
            double cx, cy, cz, c2;
            const double M = maxw(k, cx, cy, cz, c2), dMdT = M * (c2 * mc[2] - mc[3]);
            const double X = wgb + whb * RT;
            gf = rw * M;
            hf = RT * gf;
            if (wall) {
                acc[0] += X * M;
                acc[1] += rw * (X * dMdT + whb * c.R * M);
            } else {
                acc[0] += X * M;
                acc[1] += X * M * cx;
                acc[2] += X * M * cy;
                acc[3] += X * M * cz;
                acc[4] += X * dMdT + whb * c.R * M;
            }
        }
        if (wall && seed != 0.0) {
            acc[2] += wu * (u2h * gf + hf);
            acc[3] += wu * ux * gf;
            acc[4] += wu * uy * gf;
            acc[5] += wu * uz * gf;
        }
    }
    block_total(acc, std::integral_constant<int, 6>());
    if (threadIdx.x == 0) {
        double* o = a.fpar + (size_t)b * ADJ_FPAR;
        for (int j = 0; j < ADJ_FPAR; ++j) o[j] = 0.0;
        if (wall) {
            o[0] = sh[1] - sh[0] * num / (dn * dn) * dnT;
            for (int j = 0; j < 3; ++j) o[7 + j] = A * sh[3 + j];
            o[6] = a.objective == 0 ? A * sh[2]
                                    : o[7] * a.edrag[0] + o[8] * a.edrag[1] + o[9] * a.edrag[2];
        } else {
            o[1] = sh[0] / bv[0];
            for (int j = 0; j < 3; ++j) o[2 + j] = sh[1 + j] * mc[6];
            o[5] = sh[4];
        }
    }
    if (wall) {
        // through rho_w = (outflow) / (inflow of M)
        const double numb = sh[0] / dn;
        for (int k = threadIdx.x; k < c.K; k += BS) {
            const double ux = c.u[k], uy = c.u[c.Kp + k], uz = c.u[2 * c.Kp + k];
            if (leaves(k)) {
                const double un = ux * nx + uy * ny + uz * nz, wu = c.w[k] * un;
                gbar[k] = (S)(g_seed(k, un, wu, 0.5 * (ux * ux + uy * uy + uz * uz), ux, uy, uz) + numb * wu);
            }
        }
    }
}

// ------------------------------------------------------------------------------------
// cell gather 1: adjoint of phi0 from the faces where the cell is upwind, then the
// reverse of phi0 = phi_c + (x_f - u s - x_c) . L g (Eq. flux_solve_phi_phi) through the
// Venkatakrishnan limiter (Sec. 3.3 readings: minimum over faces capped at 1, eps^2
// phi_c^2 threshold) and the least-squares gradient g = sum_j M^-1 d_j (phi_j - phi_c).
// Adds the cell's own terms to its output and leaves, per slot, the neighbour's share:
// its gradient term and, if its value was Delta_max or Delta_min, that derivative.
// One warp per cell, MS >= the faces of any cell; the FP64 form takes comparisons and
// upwind signs as k_recon_d.  The share per slot (instead of the gradient's three
// components and the slot number) lets the second gather read one value a neighbour
// instead of four.
// ------------------------------------------------------------------------------------
// numerator and denominator of Venkatakrishnan's psi(d1, d2); FP32 with every rounding
// spelt out: where psi is 1 or its two candidates agree to the last bits, these decide
// which branch's derivative is taken
template <typename S>
__device__ __forceinline__ void psi_parts(S d1, S d2, S ep, S& nu, S& de) {
    if constexpr (sizeof(S) == 8) {
        const S aa = fma(d1, d1, ep), b2 = d2 + d2;
        nu = fma(d1, b2, aa);
        de = fma(d1, d2, fma(b2, d2, aa));
    } else {
        const S b2 = S(2) * d2;
        nu = __fmaf_rn(S(2) * d1, d2, __fmaf_rn(d1, d1, ep));
        de = __fadd_rn(__fmaf_rn(d1, d2, __fmaf_rn(d1, d1, __fmul_rn(b2, d2))), ep);
    }
}
template <typename S>
__device__ __forceinline__ S adj_quot(S a, S b) {
    if constexpr (sizeof(S) == 8) return quot(a, b);
    else return lim_div(a, b);
}
template <int WPB, typename S, int MS>
__global__ void __launch_bounds__(WPB * 32) k_adj_gather(Dev<double> c, AdjBufs a, AdjArr<S> r) {
    __shared__ Q4<S> s_A[WPB][MS];                // LSQ weight vector, s_ij
    __shared__ Q4<S> s_B[WPB][MS];                // x_f - x_i
    __shared__ Q4<S> s_N[WPB][MS];                // face normal
    __shared__ float4 s_F[WPB][MS];               // face normal in FP32
    __shared__ int4 s_I[WPB][MS];                 // neighbour, face, left side
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int i = blockIdx.x * WPB + w;
    if (i >= c.N) return;
    const int s0 = c.slot_off[i], ns = c.slot_off[i + 1] - s0;
    if (lane < ns) {
        const int m = s0 + lane, f = c.slot_face[m];
        s_A[w][lane] = Q4<S>{(S)c.slot_lsq[m], (S)c.slot_lsq[c.nnz + m], (S)c.slot_lsq[2 * c.nnz + m], (S)c.fs[f]};
        s_B[w][lane] = Q4<S>{(S)c.slot_d[m], (S)c.slot_d[c.nnz + m], (S)c.slot_d[2 * c.nnz + m], S(0)};
        s_N[w][lane] = Q4<S>{(S)c.slot_n[m], (S)c.slot_n[c.nnz + m], (S)c.slot_n[2 * c.nnz + m], S(0)};
        s_F[w][lane] = make_float4((float)c.slot_n[m], (float)c.slot_n[c.nnz + m], (float)c.slot_n[2 * c.nnz + m], 0.f);
        s_I[w][lane] = make_int4(c.slot_nbr[m], f, c.slot_left[m], 0);
    }
    __syncwarp();
    const S eps2 = (S)c.eps2[i];
    const int limiter = (int)a.iterp[1];
    const size_t NK = (size_t)c.N * c.Kp, FK = (size_t)c.F * c.Kp, oi = (size_t)i * c.Kp;
    for (int k = lane; k < c.K; k += 32) {
        const S ux = r.u[k], uy = r.u[c.Kp + k], uz = r.u[2 * c.Kp + k];
        unsigned up = 0;
        {
            VelF uf{};
            if constexpr (sizeof(S) == 8) uf = vel_f(c, k);
#pragma unroll
            for (int q = 0; q < MS; ++q)
                if (q < ns && adj_outflow(uf, s_F[w][q], ux, uy, uz, s_N[w][q]) == (s_I[w][q].z != 0)) up |= 1u << q;
        }
        // every load of both fields is issued before their arithmetic: the adjoint of phi0 at
        // the faces where this cell is upwind (0 elsewhere), and the neighbours' values (the
        // cell's own where there is none)
        S xf[2][MS], pn[2][MS], pcs[2], oc[2];
#pragma unroll
        for (int fd = 0; fd < 2; ++fd) {
            pcs[fd] = r.phi[fd * NK + oi + k];
            oc[fd] = r.oc[fd * NK + oi + k];
        }
#pragma unroll
        for (int q = 0; q < MS; ++q) {
            const int4 I = q < ns ? s_I[w][q] : make_int4(-1, 0, 0, 0);
            const bool u = (up >> q) & 1u;
#pragma unroll
            for (int fd = 0; fd < 2; ++fd) {
                xf[fd][q] = u ? r.fbar[fd * FK + (size_t)I.y * c.Kp + k] : S(0);
                pn[fd][q] = I.x >= 0 ? r.phi[fd * NK + (size_t)I.x * c.Kp + k] : pcs[fd];
            }
        }
#pragma unroll
        for (int fd = 0; fd < 2; ++fd) {
            const S pc = pcs[fd];
            // adjoint of phi0 gathered over the faces where this cell is upwind
            S self = S(0), sx = S(0), Gb[3] = {S(0), S(0), S(0)};
#pragma unroll
            for (int q = 0; q < MS; ++q) {
                if (q >= ns) break;
                // FP32: x is 0 where the cell is not upwind, and a divergent branch costs more
                if (sizeof(S) == 8 && !((up >> q) & 1u)) continue;
                const S x = xf[fd][q];
                const Q4<S> B = s_B[w][q];
                self += x;
                const S sq = s_A[w][q].w;
                if constexpr (sizeof(S) == 8) {
                    sx += sq * x;
                    Gb[0] += B.x * x; Gb[1] += B.y * x; Gb[2] += B.z * x;
                } else {
                    Gb[0] += (B.x - ux * sq) * x; Gb[1] += (B.y - uy * sq) * x; Gb[2] += (B.z - uz * sq) * x;
                }
            }
            S d1b = S(0), gb[3] = {S(0), S(0), S(0)};
            int slot = -1;
            if (limiter != 2) {
                if constexpr (sizeof(S) == 8) { Gb[0] -= ux * sx; Gb[1] -= uy * sx; Gb[2] -= uz * sx; }
                // forward: gradient, Delta_max/min with the slot that gave them
                S g[3] = {S(0), S(0), S(0)}, dmax = S(0), dmin = S(0);
                int amax = -1, amin = -1;
                if constexpr (sizeof(S) == 8) dmin = S(-0.0);
#pragma unroll
                for (int q = 0; q < MS; ++q) {
                    if (q >= ns) break;
                    const int j = s_I[w][q].x;
                    if (j < 0) continue;
                    const S dp = pn[fd][q] - pc;
                    const Q4<S> L = s_A[w][q];
                    g[0] += L.x * dp; g[1] += L.y * dp; g[2] += L.z * dp;
                    if constexpr (sizeof(S) == 8) {
                        const long long b = __double_as_longlong(dp);
                        if (b > __double_as_longlong(dmax)) { dmax = dp; amax = q; }
                        if ((unsigned long long)b > (unsigned long long)__double_as_longlong(dmin)) { dmin = dp; amin = q; }
                    } else {
                        if (dp > dmax) { dmax = dp; amax = q; }
                        if (dp < dmin) { dmin = dp; amin = q; }
                    }
                }
                S L = S(1);
                int lq = -1;
                S d2q = S(0);
                if (limiter == 3) {
                    L = r.lstore[fd * NK + oi + k];       // frozen: a constant
                } else if (limiter == 1) {
                    // the forward kernel's minimum: psi at the face of largest d2 (with
                    // Delta_max) and at the face of smallest d2 (with Delta_min)
                    S d2hi = S(0), d2lo = sizeof(S) == 8 ? S(-0.0) : S(0);
                    int qhi = -1, qlo = -1;
#pragma unroll
                    for (int q = 0; q < MS; ++q) {
                        if (q >= ns) break;
                        const Q4<S> B = s_B[w][q];
                        const S d2 = g[0] * B.x + g[1] * B.y + g[2] * B.z;
                        if constexpr (sizeof(S) == 8) {
                            const long long b = __double_as_longlong(d2);
                            if (b > __double_as_longlong(d2hi)) { d2hi = d2; qhi = q; }
                            if ((unsigned long long)b > (unsigned long long)__double_as_longlong(d2lo)) { d2lo = d2; qlo = q; }
                        } else {
                            if (d2 > d2hi) { d2hi = d2; qhi = q; }
                            if (d2 < d2lo) { d2lo = d2; qlo = q; }
                        }
                    }
                    const S ep = eps2 * pc * pc;
                    if (qhi >= 0) {
                        const S d1 = dmax, d2 = d2hi;
                        S nu, de;
                        psi_parts(d1, d2, ep, nu, de);
                        if (nu < de) { L = adj_quot(nu, de); lq = qhi; d2q = d2; }
                    }
                    if (qlo >= 0) {
                        const S d1 = dmin, d2 = d2lo;
                        S nu, de;
                        psi_parts(d1, d2, ep, nu, de);
                        if (nu < L * de) { L = adj_quot(nu, de); lq = qlo; d2q = d2; }
                    }
                }
                // reverse of L g
#pragma unroll
                for (int d = 0; d < 3; ++d) gb[d] = L * Gb[d];
                if (lq >= 0) {
                    const S Lb = Gb[0] * g[0] + Gb[1] * g[1] + Gb[2] * g[2];
                    const bool hi = lq >= 0 && d2q > S(0);
                    const S d2 = d2q, d1 = hi ? dmax : dmin, ep = eps2 * pc * pc;
                    S Lp2, Lself, Lp1;          // Lb times the partial derivatives of psi
                    if constexpr (sizeof(S) == 8) {
                        S nu, de;
                        psi_parts(d1, d2, ep, nu, de);
                        const S ide = quot(S(1), de), Lx = Lb * ide * ide;
                        Lp1 = Lx * ((S(2) * d1 + S(2) * d2) * de - nu * (S(2) * d1 + d2));
                        Lp2 = Lx * (S(2) * d1 * de - nu * (S(4) * d2 + d1));
                        Lself = Lx * (de - nu) * S(2) * eps2 * pc;             // through ep
                    } else {
                        // FP32: psi is homogeneous of degree 0 in (d1, d2, sqrt(ep)); its
                        // derivatives are formed from the values scaled by
                        // sigma = max(|d1|, |d2|) and divided by sigma (sigma^2 for ep), which
                        // keeps them in range.  Below sigma = 1e-30 (the far tails of the
                        // distributions) the limiter is taken as constant.
                        const S sg = fmaxf(fabsf(d1), fabsf(d2));
                        Lp1 = Lp2 = Lself = S(0);
                        if (sg > S(1e-30)) {
                            const S is = S(1) / sg, a1 = d1 * is, a2 = d2 * is, e = (ep * is) * is;
                            const S nu = a1 * a1 + e + S(2) * a1 * a2;
                            const S de = a1 * a1 + S(2) * a2 * a2 + a1 * a2 + e;
                            const S ide2 = S(1) / (de * de);
                            const S Lbs = Lb * is;
                            Lp1 = Lbs * (((S(2) * a1 + S(2) * a2) * de - nu * (S(2) * a1 + a2)) * ide2);
                            Lp2 = Lbs * ((S(2) * a1 * de - nu * (S(4) * a2 + a1)) * ide2);
                            Lself = (Lbs * ((de - nu) * ide2)) * ((S(2) * eps2 * pc) * is);
                        }
                    }
                    const Q4<S> B = s_B[w][lq];
                    gb[0] += Lp2 * B.x; gb[1] += Lp2 * B.y; gb[2] += Lp2 * B.z;
                    self += Lself;
                    const int arg = hi ? amax : amin;
                    if (arg >= 0) {
                        d1b = Lp1;
                        self -= d1b;
                        slot = arg;
                    }
                }
            }
            // reverse of the least-squares gradient: the cell's own part and the
            // neighbours' shares
            S* nb = r.nb + (size_t)fd * c.ms * NK + oi + k;
#pragma unroll
            for (int q = 0; q < MS; ++q) {
                if (q >= ns) break;
                if (s_I[w][q].x < 0) continue;
                const Q4<S> A = s_A[w][q];
                S t = A.x * gb[0] + A.y * gb[1] + A.z * gb[2];
                self -= t;
                if (slot == q) t += d1b;
                nb[(size_t)q * NK] = t;
            }
            const size_t o = fd * NK + oi + k;
            a.ophi[o] = (double)oc[fd] + (double)self;
        }
    }
}

// cell gather 2: the neighbours' shares that are this cell's, added to the output, which
// goes to dst (rows of ld doubles: the padded vector itself, or a packed one).  One warp
// per cell.
template <int WPB, typename S>
__global__ void __launch_bounds__(WPB * 32) k_adj_gather2(Dev<double> c, AdjBufs a, AdjArr<S> r, double* dst, int ld) {
    __shared__ size_t s_o[WPB][MAXF];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int i = blockIdx.x * WPB + w;
    if (i >= c.N) return;
    const int s0 = c.slot_off[i], ns = c.slot_off[i + 1] - s0;
    const size_t NK = (size_t)c.N * c.Kp, oi = (size_t)i * c.Kp;
    // offset of the share in the neighbour's record (its slot of this face)
    const int j = lane < ns ? c.slot_nbr[s0 + lane] : -1;
    const unsigned has = __ballot_sync(0xffffffffu, j >= 0);
    if (j >= 0) s_o[w][__popc(has & ((1u << lane) - 1u))] = (size_t)(a.slot_mirg[s0 + lane] - c.slot_off[j]) * NK + (size_t)j * c.Kp;
    __syncwarp();
    const int nn = __popc(has);
    for (int k = lane; k < c.K; k += 32) {
        S acc[2] = {S(0), S(0)};
        for (int q = 0; q < nn; ++q) {
            const S* nb = r.nb + s_o[w][q] + k;
            acc[0] += nb[0];
            acc[1] += nb[(size_t)c.ms * NK];
        }
        dst[(size_t)i * ld + k] = a.ophi[oi + k] + (double)acc[0];
        dst[((size_t)c.N + i) * ld + k] = a.ophi[NK + oi + k] + (double)acc[1];
    }
}

// Sum of the per-boundary-face records: out[0-5] (dR/dp)^T v or dJ/dp|_X, out[6] J,
// out[7-9] force.  One warp per value.
__global__ void __launch_bounds__(320) k_adj_params(const double* fpar, int Fb, double* out) {
    const int j = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double s = 0.0;
    for (int b = lane; b < Fb; b += 32) s += fpar[(size_t)b * ADJ_FPAR + j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) out[j] = s;
}

// ------------------------------------------------------------------------------------
// preconditioner: transposed point Gauss-Seidel sweep of the first-order implicit
// operator of Eq. implicit_mic_final_equ for the cells of one colour,
//   y_i = (r_i + sum_j (A/V_j) max(u.n_ij, 0) y_j) / D_i,
//   D_i = 1/(cfl dt_i) + 1/tau_i + sum_f (A/V_i) max(u.n_if, 0)
// (the transpose of the micro PR-SGS operator: entry (i, j) is (A/V_j) min(u.n_ji, 0)).
// One warp per cell.  DIAG writes 1/D instead, once per solve.
// ------------------------------------------------------------------------------------
template <int WPB, typename S, bool DIAG>
__global__ void __launch_bounds__(WPB * 32) k_adj_sweep(Dev<double> c, AdjBufs a, AdjArr<S> r, const int* cells, int n,
                                                        const double* b, double* y) {
    __shared__ Q4<S> s_N[WPB][MAXF], s_C[WPB][MAXF];   // scaled and unit outward normal
    __shared__ float4 s_F[WPB][MAXF];
    __shared__ int s_j[WPB][MAXF];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int t = blockIdx.x * WPB + w;
    if (t >= n) return;
    const int i = DIAG ? t : cells[t];
    const int s0 = c.slot_off[i], ns = c.slot_off[i + 1] - s0;
    if (lane < ns) {
        const int m = s0 + lane;
        const double sg = c.slot_left[m] ? 1.0 : -1.0, A = DIAG ? c.slot_AV[m] : a.slot_AVn[m];
        const double nx = sg * c.slot_n[m], ny = sg * c.slot_n[c.nnz + m], nz = sg * c.slot_n[2 * c.nnz + m];
        s_N[w][lane] = Q4<S>{(S)(A * nx), (S)(A * ny), (S)(A * nz), S(0)};
        s_C[w][lane] = Q4<S>{(S)nx, (S)ny, (S)nz, S(0)};
        s_F[w][lane] = make_float4((float)nx, (float)ny, (float)nz, 0.f);
        s_j[w][lane] = c.slot_nbr[m];
    }
    __syncwarp();
    const size_t NK = (size_t)c.N * c.Kp, oi = (size_t)i * c.Kp;
    const S base = DIAG ? (S)(1.0 / (c.cfl_imp * c.dt[i]) + 1.0 / a.tau[i]) : S(0);
    for (int k = lane; k < c.K; k += 32) {
        const S ux = r.u[k], uy = r.u[c.Kp + k], uz = r.u[2 * c.Kp + k];
        VelF uf{};
        if constexpr (sizeof(S) == 8) uf = vel_f(c, k);
        S D = base, ag = S(0), ah = S(0);
#pragma unroll 2
        for (int q = 0; q < ns; ++q) {
            const int j = s_j[w][q];
            if (!DIAG && j < 0) continue;
            if (!adj_outflow(uf, s_F[w][q], ux, uy, uz, s_C[w][q])) continue;
            const Q4<S> N = s_N[w][q];
            if (DIAG) {
                D += ux * N.x + uy * N.y + uz * N.z;
            } else {
                const S un = ux * N.x + uy * N.y + uz * N.z;
                ag += un * (S)y[(size_t)j * c.Kp + k];
                ah += un * (S)y[NK + (size_t)j * c.Kp + k];
            }
        }
        if (DIAG) {
            r.iD[oi + k] = S(1) / D;
        } else {
            const S iD = r.iD[oi + k];
            y[oi + k] = (double)(((S)b[oi + k] + ag) * iD);
            y[NK + oi + k] = (double)(((S)b[NK + oi + k] + ah) * iD);
        }
    }
}

// |u|^2 / 2 per velocity
__global__ void k_adj_u2(Dev<double> c, double* u2) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < c.Kp) u2[k] = 0.5 * (c.u[k] * c.u[k] + c.u[c.Kp + k] * c.u[c.Kp + k] + c.u[2 * c.Kp + k] * c.u[2 * c.Kp + k]);
}

// ------------------------------------------------------------------------------------
// vectors X = (phi [2][N][K], W [N][6], q [N][6]) in the packed (unpadded) layout of the
// interface <-> padded internal arrays
// ------------------------------------------------------------------------------------
// phi rows only, one warp per row (the W and q blocks are plain copies); S: the type of
// the padded side (FP32: rounded)
template <typename S>
__global__ void __launch_bounds__(256) k_adj_unpack(const double* x, size_t rows, int K, int Kp, S* phi) {
    const size_t row = blockIdx.x * (size_t)8 + (threadIdx.x >> 5);
    if (row >= rows) return;
    for (int k = threadIdx.x & 31; k < K; k += 32) phi[row * Kp + k] = (S)x[row * K + k];
}
template <typename S>
__global__ void __launch_bounds__(256) k_adj_pack(const S* phi, size_t rows, int K, int Kp, double* x) {
    const size_t row = blockIdx.x * (size_t)8 + (threadIdx.x >> 5);
    if (row >= rows) return;
    for (int k = threadIdx.x & 31; k < K; k += 32) x[row * K + k] = (double)phi[row * Kp + k];
}

// per-velocity arrays of a mixed-precision context in FP64 and back, and s_ij per slot
__global__ void k_adj_upcast(const float* src, double* dst, size_t n) {
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
        dst[t] = (double)src[t];
}
__global__ void k_adj_downcast(const double* src, float* dst, size_t n) {
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
        dst[t] = (float)src[t];
}
// *differ = 1 if any of the n doubles of a and b differ in their bits
__global__ void k_adj_differ(const double* a, const double* b, size_t n, int* differ) {
    const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (t < n && __double_as_longlong(a[t]) != __double_as_longlong(b[t])) *differ = 1;
}
__global__ void k_adj_slot_s(DevBase c, double* slot_s) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m < c.nnz) slot_s[m] = c.fs[c.slot_face[m]];
}

// ------------------------------------------------------------------------------------
// Krylov vector kernels on packed vectors of length n (deterministic: fixed grid, block
// partial sums combined in block order by k_vec_finish)
// ------------------------------------------------------------------------------------
constexpr int VEC_BS = 256, VEC_GRID = 1024;
constexpr int GM_MAX = 64;      // maximum Krylov dimension of one restart cycle

// part[b * m + j] = sum over the block's range of x . V_j, j < m (V_j = V + j * ld)
__global__ void __launch_bounds__(VEC_BS) k_vec_mdot(const double* x, const double* V, size_t ld, int m,
                                                      size_t n, double* part) {
    __shared__ double red[VEC_BS / 32];
    for (int j = 0; j < m; ++j) {
        const double* v = V + (size_t)j * ld;
        double s = 0.0;
        for (size_t t = blockIdx.x * (size_t)VEC_BS + threadIdx.x; t < n; t += (size_t)VEC_GRID * VEC_BS)
            s += x[t] * v[t];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            double tsum = red[0];
            for (int q = 1; q < VEC_BS / 32; ++q) tsum += red[q];
            part[(size_t)blockIdx.x * m + j] = tsum;
        }
        __syncthreads();
    }
}

// one warp per dot product (one thread over the 1,024 partial sums took 49 us)
__global__ void __launch_bounds__(32) k_vec_finish(const double* part, int m, double* out) {
    const int j = blockIdx.x;
    double s = 0.0;
    for (int b = threadIdx.x; b < VEC_GRID; b += 32) s += part[(size_t)b * m + j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) out[j] = s;
}

// x -= sum_j h[j] V_j  (h on the device)
__global__ void k_vec_msub(double* x, const double* V, size_t ld, int m, const double* h, size_t n) {
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x) {
        double s = x[t];
        for (int j = 0; j < m; ++j) s -= h[j] * V[(size_t)j * ld + t];
        x[t] = s;
    }
}

// y = a x + b y (a term with a zero coefficient is not read)
__global__ void k_vec_axpby(double a, const double* x, double b, double* y, size_t n) {
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
        y[t] = (a == 0.0 ? 0.0 : a * x[t]) + (b == 0.0 ? 0.0 : b * y[t]);
}

// y += sum_j c[j] V_j  (c on the device)
__global__ void k_vec_madd(double* y, const double* V, size_t ld, int m, const double* cc, size_t n) {
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x) {
        double s = y[t];
        for (int j = 0; j < m; ++j) s += cc[j] * V[(size_t)j * ld + t];
        y[t] = s;
    }
}


// ------------------------------------------------------------------------------------
// Macroscopic part of the adjoint preconditioner.  The forward iteration (Sec. 3.5)
// predicts W~ from the moments of the micro residual by the implicit macroscopic
// system (Eq. implicit_mac_equ_fin) before the micro sweeps use phi*(W~); linearised
// at a steady state it maps a residual r to
//   dW~ = L^-1 M_W r_phi,  dphi = S^-1 (r_phi + B_W dW~),  dY = M_Y dphi + r_Y,
// L the macro operator, S the micro PR-SGS operator, M_W / M_Y the moment rows of R_W /
// (R_W, R_q), B_W = dR_phi/dW.  Its transpose, applied by these kernels with the
// transposed micro sweeps, is the adjoint's preconditioner.
// ------------------------------------------------------------------------------------
// out = base + M_Y^T (yW, yq) per (cell, velocity): the weights of phi in the rows
// R_W (moments 1, u, |u|^2/2 of g; h in the energy rows) and R_q (c|c|^2/2 of g, c of h,
// c = u - U(W)); yq may be null (zero).  One warp per cell.
__global__ void __launch_bounds__(128) k_adj_momT(Dev<double> c, const double* base, const double* yW,
                                                  const double* yq, double* out) {
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * 4 + (threadIdx.x >> 5);
    if (i >= c.N) return;
    const size_t NK = (size_t)c.N * c.Kp, oi = (size_t)i * c.Kp;
    const double* a = yW + 6 * (size_t)i;
    const double* b = yq ? yq + 6 * (size_t)i : nullptr;
    const double a45 = a[4] + a[5];
    double U[3] = {0.0, 0.0, 0.0};
    if (b) {
        const double* W = c.W + 6 * (size_t)i;
        const double ir = 1.0 / W[0];
        U[0] = W[1] * ir; U[1] = W[2] * ir; U[2] = W[3] * ir;
    }
    for (int k = lane; k < c.Kp; k += 32) {
        double og = base[oi + k], oh = base[NK + oi + k];
        if (k < c.K) {
            const double ux = c.u[k], uy = c.u[c.Kp + k], uz = c.u[2 * c.Kp + k], w = c.w[k];
            const double u2h = 0.5 * (ux * ux + uy * uy + uz * uz);
            double x = a[0] + ux * a[1] + uy * a[2] + uz * a[3] + u2h * a[4], y = a45;
            if (b) {
                const double cx = ux - U[0], cy = uy - U[1], cz = uz - U[2];
                const double c2 = cx * cx + cy * cy + cz * cz;
                x += 0.5 * c2 * (cx * b[0] + cy * b[1] + cz * b[2]);
                y += cx * b[3] + cy * b[4] + cz * b[5];
            }
            og += w * x;
            oh += w * y;
        }
        out[oi + k] = og;
        out[NK + oi + k] = oh;
    }
}

// ---- transposed macro PR-SGS ----------------------------------------------------------
// Point update of cell j on L^T: y_j = D_j^-1 (b_j - sum_i (J(W_j; n)^T y_i - c r y_i)) over
// the interior neighbours i, n the normal out of i scaled by c = A_f / (2 V_i) (the forward
// operator's coefficient of dW_j in row i, transposed) and J^T y the gradient of
// y . G(W; n) (Eq. implicit_mac_equ_euler_flux; p = (2/5)(rho E - rho |U|^2 / 2)).  With
//   t = U.n - c r,  e = (rho E + p)/rho,  e_r = E_rot/rho,
//   A = y_0 + y_m.U + e y_4 + e_r y_5,  B = y_m.n + y_4 U.n  (m: the momentum components)
// a face adds (t y_0 - U.n A, t y_m + n A, t y_4, t y_5) and the sum of B adds
// 0.2 |U|^2, -0.4 U and 0.4 of itself at the end: 20 FP64 operations a face, with all that
// depends on the state formed once per state, against some 110 with the divisions of
// J(W_j) in every face of every phase.  Layout and threads as the forward solve's
// (macro_point): y [p][8] by colour position; constants mC [8][p]: U, 0.2 |U|^2, e, e_r,
// 1/D, 1/(D + 1/(Z tau)); slots mS [5][ms][p]: n, U.n, t.
// A phase of 1,478 cells took 18.1 us.
__global__ void __launch_bounds__(128) k_adj_macro_prep(Dev<double> c, const int* col_cell, const double* tau,
                                                        double* mC, double* mS) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= c.N) return;
    const int j = col_cell[p];
    const size_t N = (size_t)c.N;
    const double* W = c.W + 6 * (size_t)j;
    const double ir = 1.0 / W[0], U[3] = {W[1] * ir, W[2] * ir, W[3] * ir};
    const double U2 = U[0] * U[0] + U[1] * U[1] + U[2] * U[2];
    const double pr = 0.4 * (W[4] - 0.5 * W[0] * U2);
    double D = 1.0 / (c.cfl_imp * c.dt[j]);
    const double hv = 0.5 / c.vol[j];
    const int s0 = c.slot_off[j];
    for (int m = s0; m < c.slot_off[j + 1]; ++m) {
        const int f = c.slot_face[m], i = c.slot_nbr[m];
        D += hv * c.fa[f] * c.rf[f];
        const double cij = i >= 0 ? 0.5 * c.fa[f] / c.vol[i] : 0.0, sg = c.slot_left[m] ? -cij : cij;
        double* S = mS + (size_t)(m - s0) * N + p;
        double Un = 0.0;
        for (int d = 0; d < 3; ++d) {
            const double n = sg * c.fn[(size_t)d * c.F + f];
            S[(size_t)d * c.ms * N] = n;
            Un += U[d] * n;
        }
        S[(size_t)3 * c.ms * N] = Un;
        S[(size_t)4 * c.ms * N] = Un - cij * c.rf[f];
    }
    for (int d = 0; d < 3; ++d) mC[d * N + p] = U[d];
    mC[3 * N + p] = 0.2 * U2;
    mC[4 * N + p] = (W[4] + pr) * ir;
    mC[5 * N + p] = W[5] * ir;
    mC[6 * N + p] = 1.0 / D;
    mC[7 * N + p] = 1.0 / (D + 1.0 / (c.Z * tau[j]));
}

template <int L>
__global__ void __launch_bounds__(MACRO_BS) k_adj_macro_sweepT(const __grid_constant__ DevBase c, const int* col_cell,
                                                               int lo, int n, const double* mC, const double* mS,
                                                               const double* b, double* y) {
    const int t0 = (blockIdx.x * blockDim.x + threadIdx.x) / L;
    if (t0 >= n) return;                          // whole lane group
    const int g = (int)(threadIdx.x % L), p = lo + t0;
    const size_t N = (size_t)c.N;
    double C[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) C[q] = mC[q * N + p];
    constexpr int U = L >= 4 ? 2 : 4;
    int j[U];
    double s[U][5];
    auto load_slots = [&](int q0) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int q = q0 + u * L;
            j[u] = q < c.ms ? c.mNbr[q * N + p] : -1;
            if (j[u] >= 0)
#pragma unroll
                for (int d = 0; d < 5; ++d) s[u][d] = mS[(size_t)(d * c.ms + q) * N + p];
        }
    };
    load_slots(g);
    double o[6] = {0, 0, 0, 0, 0, 0}, B = 0.0;    // o: the face terms less b
    if (g == 0) {
        const double* bp = b + 6 * (size_t)col_cell[p];
#pragma unroll
        for (int q = 0; q < 6; ++q) o[q] = -bp[q];
    }
    pdl_wait();
    pdl_launch_dependents();
    for (int q0 = g;;) {
        double Y[U][8];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (j[u] >= 0) macro_load(y + 8 * (size_t)j[u], Y[u]);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (j[u] >= 0) {
                const double* v = Y[u];
                const double A = fma(v[1], C[0], fma(v[2], C[1], fma(v[3], C[2], fma(v[4], C[4], fma(v[5], C[5], v[0])))));
                B = fma(v[1], s[u][0], fma(v[2], s[u][1], fma(v[3], s[u][2], fma(v[4], s[u][3], B))));
                o[0] = fma(s[u][4], v[0], fma(-s[u][3], A, o[0]));
                o[1] = fma(s[u][4], v[1], fma(s[u][0], A, o[1]));
                o[2] = fma(s[u][4], v[2], fma(s[u][1], A, o[2]));
                o[3] = fma(s[u][4], v[3], fma(s[u][2], A, o[3]));
                o[4] = fma(s[u][4], v[4], o[4]);
                o[5] = fma(s[u][4], v[5], o[5]);
            }
        q0 += U * L;
        if (q0 >= c.ms) break;
        load_slots(q0);
    }
    group_sum6<L>(o);
    if constexpr (L > 1) {
        const int base = (threadIdx.x & 31) & ~(L - 1);
        const unsigned mask = ((1u << L) - 1u) << base;
#pragma unroll
        for (int f = 1; f < L; f <<= 1) B += __shfl_xor_sync(mask, B, f);
    }
    if (g != 0) return;
    const double r0 = fma(-C[3], B, -o[0]), B4 = 0.4 * B;
    const double r1 = fma(C[0], B4, -o[1]), r2 = fma(C[1], B4, -o[2]), r3 = fma(C[2], B4, -o[3]);
    const double r4 = -o[4] - B4, r5 = -o[5];
    double2* P = reinterpret_cast<double2*>(y + 8 * (size_t)p);
    __stcg(P, make_double2(r0 * C[6], r1 * C[6]));
    __stcg(P + 1, make_double2(r2 * C[6], r3 * C[6]));
    __stcg(P + 2, make_double2(r4 * C[6], r5 * C[7]));
}

// the iterate by cell [N][6] from its records by colour position
__global__ void k_adj_macro_out(DevBase c, const double* y, double* o) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= c.N) return;
    const double* r = y + 8 * (size_t)c.cell_pos[i];
    for (int q = 0; q < 6; ++q) o[6 * (size_t)i + q] = r[q];
}

}  // namespace rk
