// Synthetic (macroscopic) equations of GSIS on 1-D and 2-D meshes (Sections 2.2, 3 and 5).
//
//  macro_from_fields   W = conservative variables of a field record, and the primitive ones
//  macro_grad          least-squares gradients, Venkatakrishnan limiters and (order 2) the
//                      reconstructed face values of every cell (the stencil of the sweep)
//  macro_flux          three kinds of thread blocks in one launch: the flux and the Gamma of
//                      every interior face; the flux through every boundary face (walls: an
//                      equilibrium leaving at the cell state against the diffuse wall, as
//                      discrete velocity and direction sums; far field: Rusanov plus NSF
//                      against the free stream); the sources of every cell and their
//                      Jacobian's coefficients
//  macro_hot           face high-order terms of Eq. (getHoTs), projected on the face normal:
//                      kinetic stress and heat fluxes averaged to the face minus the NSF
//                      values of the kinetic state; boundary terms = kinetic minus
//                      macroscopic boundary flux
//  macro_residual      R = -(1/V) sum (F_c + F_v) S + Q (Eq. delta_macro, right-hand side),
//                      the implicit diagonal D (with the exact local Jacobian of the energy
//                      sources) and its inverse, the first relaxation sweep D dW = R, and
//                      ||R||_2 with the stop flag (its last block)
//  macro_jacobi        one further point-relaxation sweep of
//                      D dW_i + (1/(2V)) sum_j (dF_j - Gamma dW_j) S = R_i
//                      in the gas-energy form; the last one adds dW to W
// (kinetic_bflux, the kinetic boundary fluxes, and sync, the update of f by the synthetic
// solution, are in kernels.cu.)
//
// Every kernel of the inner loop returns at once when the solve's stop flag is set,
// so a fixed launch sequence can run past convergence without changing W.
//
// What bounds these kernels is the number of FP64 instructions on the longest chain (64 to
// 76 cycles each, see fp64.cuh), then the launches (about 1 us each) and the chains of
// dependent loads; the data (a few MB) stay in L2.  Hence: no divisions by geometry or
// model constants (stored as reciprocals, in the compute type, so that the FP32 path
// converts nothing), one lane per variable or row of a cell where few warps are in flight,
// face fluxes once per face, and the relaxation reads its neighbours' flux increments as
// vectors F_a that the neighbour formed once, not once per adjacent face.
// Per inner iteration (six sweeps, a GSIS iteration less its kinetic part over 100): 20 000
// cells, mixed schedule 307 -> 72 us; 2 048 cells, FP64 209 -> 61 us, mixed 112 -> 40 us;
// 800 cells in 1-D, FP64, order 2, 174 -> 43 us.
#include <algorithm>
#include <cmath>

#include "gsis_impl.cuh"
#include "fp64.cuh"

namespace gsis {

namespace {

constexpr double PI = 3.14159265358979323846;

// The kernels of the inner loop are launched before their predecessor in the stream has ended
// (launch_after), so that only the wait for its last block remains of the time between two
// kernels; a kernel reads and writes nothing before every block of its predecessor has ended
// and its writes are visible.  Every thread waits, so that the end of a kernel implies the end
// of all before it.  300 inner iterations: 800 cells FP64 14.4 -> 13.7 ms, 2 048 cells FP64
// 22.5 -> 22.1, 20 000 cells mixed 17.2 -> 16.9.  With the next kernel's blocks let in when
// those of the current one have started (griddepcontrol.launch_dependents) these took 14.8,
// 28.6 and 19.4 ms, and halfway through the kernels 13.8, 22.0 and 18.2.
// The kernels take plain pointers and hand them to a body that holds the __restrict__: a load
// through a __restrict__ argument of the kernel itself may be moved above the wait.
__device__ __forceinline__ void wait_for_previous() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename... P, typename... A>
cudaError_t launch_after(cudaStream_t s, void (*kernel)(P...), int grid, int block, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// Device functions are templates on the compute type R (double for the plain FP64 path,
// float for the FP32 path's residual evaluation).
template <typename R>
__device__ __forceinline__ const MacroReal<R> &real(const MacroGeom &g) {
    if constexpr (sizeof(R) == 8) return g.d;
    else return g.f;
}

// mu = p_t tau
template <typename R>
__device__ __forceinline__ R viscosity(R T_t, const MacroReal<R> &c) { return c.mu0 * pow_r(T_t, c.omega); }
template <typename R>
__device__ __forceinline__ R sound_speed(R T_t) { return sqrt_r(R(5.0 / 3.0) * T_t); }
template <typename R>
__device__ __forceinline__ R absorption(R rho, const MacroReal<R> &c) { return c.dens ? c.ik * rho : c.ik; }
template <typename R>
__device__ __forceinline__ R vib_e(R T, const ModelDev &m, const MacroReal<R> &c) {
    return m.dv_T ? vib_energy<R>(m, T) : c.half_dv * T;
}

// base = A^-1 diag(5, d_r, d_v) at d_v(T_v) of the face (Eq. NSF_thermal_conductivities,
// kappa_gas = mu/2 base), or the model's constant one
template <typename R>
__device__ void kappa_at(const ModelDev &m, const MacroReal<R> &c, double Tv, R (&B)[3][3]) {
    if (!m.dv_T) {
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) B[a][b] = c.base[a * 3 + b];
        return;
    }
    double A[9], D[9];
    const double dv = dv_at(m, Tv);
    relaxation_matrix_at(m, dv, A);
    kappa_base(A, m.d_r, dv, D);
    for (int k = 0; k < 9; ++k) B[k / 3][k % 3] = R(D[k]);
}

template <int DIM>
__device__ __forceinline__ void primitive(const double *W, const ModelDev &m, const MacroReal<double> &c, double *q) {
    constexpr int E = 1 + DIM;
    const double rho = W[0], ir = rcp_r(rho);
    double ke = 0.0;
    q[0] = rho;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        q[1 + a] = W[1 + a] * ir;
        ke = fma(q[1 + a], W[1 + a], ke);
    }
    q[E] = (W[E] - W[E + 3] - W[E + 1] - W[E + 2] - 0.5 * ke) * ((2.0 / 3.0) * ir);
    q[E + 1] = W[E + 1] * (c.i_half_dr * ir);
    q[E + 2] = m.dv_T ? vib_temperature<double>(m, W[E + 2] * ir) : W[E + 2] * (c.i_half_dv * ir);
    q[E + 3] = W[E + 3];
}

template <int DIM>
__device__ __forceinline__ void prim_to_W(const double *q, const ModelDev &m, double *W) {
    constexpr int E = 1 + DIM;
    const double rho = q[0];
    double uu = 0.0;
    for (int a = 0; a < DIM; ++a) uu += q[1 + a] * q[1 + a];
    const double er = 0.5 * m.d_r * rho * q[E + 1], ev = rho * vib_energy<double>(m, q[E + 2]);
    W[0] = rho;
    for (int a = 0; a < DIM; ++a) W[1 + a] = rho * q[1 + a];
    W[E] = 1.5 * rho * q[E] + 0.5 * rho * uu + er + ev + q[E + 3];
    W[E + 1] = er;
    W[E + 2] = ev;
    W[E + 3] = q[E + 3];
}

// One side of a face: the convected variables U (rho, m, gas energy, e_r, e_v), their flux
// F_c . n of Eq. (macroscopic_equation) and |u_n| + c_s.  e_R has no convective flux.
template <typename R, int DIM>
__device__ __forceinline__ R face_side(const R *q, const R *n, const ModelDev &m, const MacroReal<R> &c, R *U, R *F) {
    constexpr int E = 1 + DIM;
    const R rho = q[0];
    R un = R(0), ke = R(0);
    U[0] = rho;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        U[1 + a] = rho * q[1 + a];
        un = fma(q[1 + a], n[a], un);
        ke = fma(U[1 + a], q[1 + a], ke);
    }
    const R p = rho * q[E];
    U[E + 1] = c.half_dr * rho * q[E + 1];
    U[E + 2] = rho * vib_e(q[E + 2], m, c);
    U[E] = fma(R(1.5), p, fma(R(0.5), ke, U[E + 1] + U[E + 2]));
    F[0] = rho * un;
#pragma unroll
    for (int a = 0; a < DIM; ++a) F[1 + a] = fma(U[1 + a], un, p * n[a]);
    F[E] = un * (U[E] + p);
    F[E + 1] = un * U[E + 1];
    F[E + 2] = un * U[E + 2];
    return fabs(un) + sound_speed(q[E]);
}

// Rusanov flux times `scale`: average of the two fluxes minus half the largest |u_n| + c_s
// times the jump of the convected variables (gas energy, not e_R)
template <typename R, int DIM>
__device__ __forceinline__ void rusanov(const R *qL, const R *qR, const R *n, R scale, const ModelDev &m,
                                        const MacroReal<R> &c, R *F) {
    constexpr int E = 1 + DIM;
    R UL[E + 3], UR[E + 3], FL[E + 3], FR[E + 3];
    const R lL = face_side<R, DIM>(qL, n, m, c, UL, FL), lR = face_side<R, DIM>(qR, n, m, c, UR, FR);
    const R lam = max_pos(lL, lR), h = R(0.5) * scale;
#pragma unroll
    for (int k = 0; k < E + 3; ++k) F[k] = h * fma(lam, UL[k] - UR[k], FL[k] + FR[k]);
    F[E + 3] = R(0);
}

// Venkatakrishnan's limiter function phi_V = num / den
template <typename R>
__device__ __forceinline__ void venkat(R d1, R d2, R eps2, R &num, R &den) {
    const R t = d1 + d2;
    num = fma(d1, t + d2, eps2);
    den = fma(d1, t, fma(d2 + d2, d2, eps2));
}

}  // namespace

// ------------------------------------------------------------------ conversions (FP64)
// q [nc][NVM] in FP64, and its rounding qf where the FP32 path reads it (else null)
template <int DIM>
__global__ void k_macro_from_fields(int n_cells, ModelDev m, const double *__restrict__ F, double *__restrict__ W,
                                    double *__restrict__ q, float *__restrict__ qf) {
    constexpr int NV = DIM + 5, E = 1 + DIM;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_cells) return;
    const double *r = F + (size_t)i * NF;
    double x[NV];
    x[0] = r[0];
    for (int a = 0; a < DIM; ++a) x[1 + a] = r[1 + a];
    x[E] = r[4];
    x[E + 1] = r[5];
    x[E + 2] = r[6];
    const double TR = r[7];
    x[E + 3] = 4.0 * m.sigma_R * TR * TR * TR * TR;
    prim_to_W<DIM>(x, m, W + (size_t)i * NVM);
    for (int v = 0; v < NV; ++v) {
        q[(size_t)i * NVM + v] = x[v];
        if (qf) qf[(size_t)i * NVM + v] = fp64::narrow(x[v]);
    }
}

// fac: null, or the factor of k_macro_mass that W is scaled by
template <int DIM>
__global__ void k_macro_fields_from_W(int n_cells, ModelDev m, MacroReal<double> c, const double *__restrict__ W,
                                      const double *__restrict__ fac, double *__restrict__ F) {
    constexpr int NV = DIM + 5, E = 1 + DIM;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_cells) return;
    double w[NV], q[NV];
    const double s = fac ? *fac : 1.0;
    for (int v = 0; v < NV; ++v) w[v] = s * W[(size_t)i * NVM + v];
    primitive<DIM>(w, m, c, q);
    double *r = F + (size_t)i * NF;
    for (int k = 0; k < NF; ++k) r[k] = 0.0;
    r[0] = q[0];
    for (int a = 0; a < DIM; ++a) r[1 + a] = q[1 + a];
    r[4] = q[E];
    r[5] = q[E + 1];
    r[6] = q[E + 2];
    r[7] = sqrt_r(sqrt_r(fmax(q[E + 3], 0.0) / (4.0 * m.sigma_R)));
}

// ------------------------------------------------------------------ gradients and limiters
// Eight lanes per cell, lane v = primitive variable v: q [nc][NVM] -> grad [nc][MGS][NVM]
// and, at order 2, the limited reconstruction at every interior face of the cell,
// rec [nc][MAXF][NVM].  The limiter's minimum over the faces is taken at the largest and the
// most negative Delta_2 (phi_V falls beyond Delta_1 / 4 and exceeds 1 below Delta_1 / 2), and
// in FP64 the smaller of the two quotients is found without dividing (their terms are positive).
template <typename R, int DIM, int ORDER>
__device__ __forceinline__ void k_macro_grad_body(MacroGeom g, const MacroState *__restrict__ st, R *__restrict__ grad, R *__restrict__ rec) {
    constexpr int NV = DIM + 5, MS = Lay<DIM>::MAXS, LW = Lay<DIM>::LW;
    if (st && st->done) return;
    const MacroReal<R> &c = real<R>(g);
    const int t = blockIdx.x * blockDim.x + threadIdx.x, i = t / NVM, v = t % NVM;
    if (i >= g.n_cells || v >= NV) return;
    const R qi = c.q[(size_t)i * NVM + v];
    R gr[DIM], hi = R(0), lo = -R(0);
#pragma unroll
    for (int a = 0; a < DIM; ++a) gr[a] = R(0);
    const int4 info = g.info[i];
    const int *stn = g.stn + (size_t)i * MS;
    const R *lw = c.lsq + (size_t)i * MS * LW;
    // two entries at a time: entries past the end hold cell 0 and zero weights
    for (int k = 0; k < info.y; k += 2) {
        const R q0 = c.q[(size_t)stn[k] * NVM + v], q1 = c.q[(size_t)stn[k + 1] * NVM + v];
        const R d0 = q0 - qi, d1 = q1 - qi;
#pragma unroll
        for (int a = 0; a < DIM; ++a) gr[a] = fma(lw[k * LW + a], d0, gr[a]);
        if (k + 1 < info.y) {
#pragma unroll
            for (int a = 0; a < DIM; ++a) gr[a] = fma(lw[(k + 1) * LW + a], d1, gr[a]);
        }
        if (ORDER == 2 && k < info.z) {
            hi = max_pos(hi, d0);
            lo = min_neg(lo, d0);
            if (k + 1 < info.z) {
                hi = max_pos(hi, d1);
                lo = min_neg(lo, d1);
            }
        }
    }
#pragma unroll
    for (int a = 0; a < DIM; ++a) grad[((size_t)i * MGS + a) * NVM + v] = gr[a];
    if constexpr (ORDER == 2) {
        R d2[MAXF], h2 = R(0), l2 = -R(0);
#pragma unroll
        for (int k = 0; k < MAXF; ++k) {
            d2[k] = R(0);
            if (g.nb[i * MAXF + k] < 0) continue;
            const R *dx = c.cdx + ((size_t)i * MAXF + k) * MGS;
#pragma unroll
            for (int a = 0; a < DIM; ++a) d2[k] = fma(gr[a], dx[a], d2[k]);
            h2 = max_pos(h2, d2[k]);
            l2 = min_neg(l2, d2[k]);
        }
        const R eps2 = c.eps2[i];
        R nh, dh, nl, dl;
        venkat(hi, h2, eps2, nh, dh);       // h2 = 0: num = den, phi = 1
        venkat(lo, l2, eps2, nl, dl);
        R phi;
        if constexpr (sizeof(R) == 8) {
            const bool low = nl * dh < nh * dl;
            const R num = low ? nl : nh, den = low ? dl : dh;
            phi = num < den ? num * rcp_r(den) : R(1);
        } else {
            phi = fmin(fmin(R(1), nh < dh ? nh / dh : R(1)), nl < dl ? nl / dl : R(1));
        }
#pragma unroll
        for (int k = 0; k < MAXF; ++k)
            if (g.nb[i * MAXF + k] >= 0) rec[((size_t)i * MAXF + k) * NVM + v] = fma(phi, d2[k], qi);
    }
}
template <typename R, int DIM, int ORDER>
__global__ void __launch_bounds__(128) k_macro_grad(MacroGeom g, const MacroState *st, R *grad, R *rec) {
    wait_for_previous();
    k_macro_grad_body<R, DIM, ORDER>(g, st, grad, rec);
}

// ------------------------------------------------------------------ face fluxes
namespace {

// NSF terms of an interior face on its normal: sn = sigma . n (DIM), qn = q . n of the
// translational, rotational and vibrational modes and of the photons (4); pf the
// face-average state.  Eqs. (NSF_constitutive) and (NSF_thermal_conductivities) with the
// face gradient = average of the cells' least-squares gradients with the component along
// x_j - x_i replaced by the difference quotient; the scalars need its normal component only.
template <typename R, int DIM>
__device__ __forceinline__ void nsf_normal(const MacroGeom &g, const ModelDev &m, const R *fg16, int i, int j,
                                           const R *__restrict__ grad, R *pf, R &mu, R &irho, R &kR, R *sn, R *qn) {
    constexpr int E = 1 + DIM, NV = DIM + 5;
    const MacroReal<R> &c = real<R>(g);
    const R *n = fg16, *t = fg16 + 3, *mh = fg16 + 6;
    const R invd = fg16[9], tnd = fg16[10];
    const R *qi = c.q + (size_t)i * NVM, *qj = c.q + (size_t)j * NVM;
    const R *gi = grad + (size_t)i * MGS * NVM, *gj = grad + (size_t)j * MGS * NVM;
    R jump[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const R a = qi[v], b = qj[v];
        pf[v] = R(0.5) * (a + b);
        jump[v] = b - a;
    }
    R gu[DIM][DIM];       // gu[a][b] = d u_b / d x_a
#pragma unroll
    for (int b = 0; b < DIM; ++b) {
        R s[DIM], along = R(0);
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            s[a] = R(0.5) * (gi[a * NVM + 1 + b] + gj[a * NVM + 1 + b]);
            along = fma(t[a], s[a], along);
        }
        const R d = fma(jump[1 + b], invd, -along);
#pragma unroll
        for (int a = 0; a < DIM; ++a) gu[a][b] = fma(t[a], d, s[a]);
    }
    R gn[4];              // normal derivatives of T_t, T_r, T_v, e_R
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        gn[k] = tnd * jump[E + k];
#pragma unroll
        for (int a = 0; a < DIM; ++a) gn[k] = fma(mh[a], gi[a * NVM + E + k] + gj[a * NVM + E + k], gn[k]);
    }
    R base[3][3];
    kappa_at<R>(m, c, m.dv_T ? to_double(pf[E + 2]) : 0.0, base);
    mu = viscosity(pf[E], c);
    R div = R(0);
#pragma unroll
    for (int a = 0; a < DIM; ++a) div += gu[a][a];
    div *= R(2.0 / 3.0);
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        R s = -div * n[a];
#pragma unroll
        for (int b = 0; b < DIM; ++b) s = fma(gu[a][b] + gu[b][a], n[b], s);
        sn[a] = -mu * s;
    }
    const R hm = R(-0.5) * mu;
#pragma unroll
    for (int md = 0; md < 3; ++md) qn[md] = hm * fma(base[md][0], gn[0], fma(base[md][1], gn[1], base[md][2] * gn[2]));
    irho = rcp_r(pf[0]);
    kR = c.dens ? c.kR0 * irho : c.kR0;
    qn[3] = -kR * gn[3];
}

// Far-field boundary flux: Rusanov against the free stream plus NSF terms over the
// distance from the cell centre to the face
template <typename R, int DIM>
__device__ void farfield_flux(const MacroGeom &g, const ModelDev &m, int b, const R *qc, R *F) {
    constexpr int E = 1 + DIM;
    const MacroReal<R> &c = real<R>(g);
    const double *P = g.patch_state + (size_t)g.bf_patch[b] * 8;
    R base[3][3];
    kappa_at<R>(m, c, m.dv_T ? 0.5 * (to_double(qc[E + 2]) + P[6]) : 0.0, base);   // at the face's T_v
    const R *bg = c.bgeo + (size_t)b * 8;
    R n[DIM];
    for (int a = 0; a < DIM; ++a) n[a] = bg[a];
    const R idn = bg[4];
    R qf[DIM + 5];
    qf[0] = R(P[0]);
    for (int a = 0; a < DIM; ++a) qf[1 + a] = R(P[1 + a]);
    qf[E] = R(P[4]);
    qf[E + 1] = R(P[5]);
    qf[E + 2] = R(P[6]);
    qf[E + 3] = R(4.0 * m.sigma_R * P[7] * P[7] * P[7] * P[7]);
    rusanov<R, DIM>(qc, qf, n, R(1), m, c, F);
    const R mu = viscosity(R(0.5) * (qc[E] + qf[E]), c);
    R du[DIM], dun = R(0);
    for (int a = 0; a < DIM; ++a) {
        du[a] = qf[1 + a] - qc[1 + a];
        dun += n[a] * du[a];
    }
    R sn[DIM], snu = R(0);
    for (int a = 0; a < DIM; ++a) {
        sn[a] = -mu * idn * (du[a] + (dun * R(1.0 / 3.0)) * n[a]);
        snu += sn[a] * R(0.5) * (qf[1 + a] + qc[1 + a]);
    }
    const R dT[3] = {qf[E] - qc[E], qf[E + 1] - qc[E + 1], qf[E + 2] - qc[E + 2]};
    R qm[3];
    for (int md = 0; md < 3; ++md) {
        R s = R(0);
        for (int nn = 0; nn < 3; ++nn) s += R(0.5) * mu * base[md][nn] * dT[nn];
        qm[md] = -s * idn;
    }
    const R kR = c.dens ? c.kR0 * rcp_r(qc[0]) : c.kR0;
    const R qR = -(qf[E + 3] - qc[E + 3]) * kR * idn;
    for (int a = 0; a < DIM; ++a) F[1 + a] += sn[a];
    F[E] += snu + (qm[0] + qm[1] + qm[2]) + qR;
    F[E + 1] += qm[1];
    F[E + 2] += qm[2];
    F[E + 3] += qR;
}

constexpr int MF_NT = 128;            // threads of a flux CTA
constexpr int MF_FACES = MF_NT / 2;   // interior faces of one: half the threads take each part

// sum over the CTA of each of N values per thread, valid in thread 0
template <int N, typename R>
__device__ __forceinline__ void cta_sum(R (&x)[N], R (&buf)[MF_NT / 32][N]) {
#pragma unroll
    for (int k = 0; k < N; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x[k] += __shfl_xor_sync(0xffffffffu, x[k], o);
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int k = 0; k < N; ++k) buf[threadIdx.x >> 5][k] = x[k];
    __syncthreads();
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < N; ++k) x[k] = (buf[0][k] + buf[1][k]) + (buf[2][k] + buf[3][k]);
}

__device__ __forceinline__ double gauss(double mB, double c2) { return fp64::exp2n(mB * fp64::EXP_SCALE, c2); }
__device__ __forceinline__ float gauss(float mB, float c2) { return expf(mB * c2); }

// Flux through boundary face b (one CTA).  Walls: outgoing molecules in equilibrium at the
// cell state, incoming ones the diffuse wall Maxwellian with the density that zeroes the
// mass flux; photons leave isotropically (e_R / 4 pi) and enter black-body
// (sigma_R T_w^4 / pi).  All four planes of the cell's equilibrium are multiples of F0, so
// three kinds of sums give every row; the wall's own sums (unit density) and the direction
// sums do not change and are kept in g.binc (k_macro_binc).
template <typename R, int DIM>
__device__ void boundary_face(const MacroGeom &g, const ModelDev &m, const QuadD &vq, int b, double *__restrict__ bflux) {
    constexpr int NV = DIM + 5, E = 1 + DIM, MH = 3 - DIM, NS = DIM + 4, N = DIM + 2;
    const MacroReal<R> &c = real<R>(g);
    __shared__ R buf[MF_NT / 32][N];
    const int cell = g.bf_cell[b], patch = g.bf_patch[b], pk = g.patch_kind[patch];
    R qc[NV];
    for (int k = 0; k < NV; ++k) qc[k] = c.q[(size_t)cell * NVM + k];
    double *out = bflux + (size_t)b * NVM;
    const R *bg = c.bgeo + (size_t)b * 8;
    R n[DIM];
    for (int a = 0; a < DIM; ++a) n[a] = bg[a];
    if (pk != 0) {
        if (threadIdx.x != 0) return;
        R F[NV];
        if (pk == 2) {   // mirror plane: Rusanov against the cell state with its normal velocity reversed
            R qm[NV], un = R(0);
            for (int a = 0; a < DIM; ++a) un += qc[1 + a] * n[a];
            for (int k = 0; k < NV; ++k) qm[k] = qc[k];
            for (int a = 0; a < DIM; ++a) qm[1 + a] = qc[1 + a] - R(2) * un * n[a];
            rusanov<R, DIM>(qc, qm, n, R(1), m, c, F);
        } else {
            farfield_flux<R, DIM>(g, m, b, qc, F);
        }
        for (int k = 0; k < NV; ++k) out[k] = to_double(F[k]);
        return;
    }
    const R Tt = qc[E], mB = R(-0.5) * rcp_r(Tt);
    R acc[N];
#pragma unroll
    for (int k = 0; k < N; ++k) acc[k] = R(0);
    for (int v = threadIdx.x; v < vq.n; v += MF_NT) {
        R xi[DIM], xn = R(0);
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            xi[a] = c.vx[a * vq.n_pad + v];
            xn = fma(xi[a], n[a], xn);
        }
        if (is_neg(xn)) continue;
        R c2 = R(0), x2 = R(0);
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            const R d = xi[a] - qc[1 + a];
            c2 = fma(d, d, c2);
            x2 = fma(xi[a], xi[a], x2);
        }
        const R wf = c.vw[v] * xn * gauss(mB, c2);
        acc[0] += wf;
#pragma unroll
        for (int a = 0; a < DIM; ++a) acc[1 + a] = fma(wf, xi[a], acc[1 + a]);
        acc[1 + DIM] = fma(wf, x2, acc[1 + DIM]);
    }
    cta_sum<N>(acc, buf);
    if (threadIdx.x != 0) return;
    const double *in = g.binc + (size_t)b * BINC;
    // F0 = rho (2 pi T)^(-DIM/2) exp(-c^2 / 2T)
    const R i2piT = rcp_r(R(2.0 * PI) * Tt);
    const R Ac = qc[0] * (DIM == 2 ? i2piT : sqrt_r(i2piT));
    const R hr = c.half_dr * qc[E + 1], hv = vib_e(qc[E + 2], m, c);
    R r[NS];
    r[0] = Ac * acc[0];
#pragma unroll
    for (int a = 0; a < DIM; ++a) r[1 + a] = Ac * acc[1 + a];
    r[E] = fma(R(0.5) * Ac, acc[1 + DIM], fma(R(0.5 * MH), Tt, hr + hv) * r[0]);
    r[E + 1] = hr * r[0];
    r[E + 2] = hv * r[0];
    const double rw = -to_double(r[0]) * in[NS + 2];   // in[NS + 2] = 1 / in[0]
    const double FR = fma(to_double(qc[E + 3]), in[NS], in[NS + 1]);
    for (int k = 0; k < NS; ++k) {
        const double x = fma(rw, in[k], to_double(r[k]));
        out[k] = k == E ? x + FR : x;
    }
    out[E + 3] = FR;
}

}  // namespace

// The constant sums of every wall face: rows of the unit-density wall Maxwellian over the
// entering velocities (NS), sum of the leaving directions over 4 pi, black-body flux of the
// entering ones, reciprocal of the first.  Runs when the velocity sets are set.
template <int DIM>
__global__ void __launch_bounds__(MF_NT) k_macro_binc(MacroGeom g, ModelDev m, QuadD vq, QuadD oq,
                                                      double *__restrict__ binc) {
    constexpr int E = 1 + DIM, NS = DIM + 4, MH = 3 - DIM;
    __shared__ double buf[MF_NT / 32][NS + 2];
    const int b = blockIdx.x, patch = g.bf_patch[b];
    if (g.patch_kind[patch] != 0) return;
    const double *P = g.patch_state + (size_t)patch * 8, *n = g.d.bgeo + (size_t)b * 8;
    const double Tw = P[4], evw = vib_energy<double>(m, Tw);
    double acc[NS + 2];
    for (int k = 0; k < NS + 2; ++k) acc[k] = 0.0;
    for (int v = threadIdx.x; v < vq.n; v += MF_NT) {
        double xi[DIM], xn = 0.0, x2 = 0.0, c2 = 0.0;
        for (int a = 0; a < DIM; ++a) {
            xi[a] = vq.x[a * vq.n_pad + v];
            xn += xi[a] * n[a];
            x2 += xi[a] * xi[a];
            c2 += (xi[a] - P[1 + a]) * (xi[a] - P[1 + a]);
        }
        if (xn > 0.0) continue;
        const double f0 = pow(2.0 * PI * Tw, -0.5 * DIM) * exp(-0.5 * c2 / Tw), wf = vq.w[v] * xn;
        acc[0] += wf * f0;
        for (int a = 0; a < DIM; ++a) acc[1 + a] += wf * f0 * xi[a];
        acc[E] += wf * (0.5 * x2 + 0.5 * MH * Tw + 0.5 * m.d_r * Tw + evw) * f0;
        acc[E + 1] += wf * 0.5 * m.d_r * Tw * f0;
        acc[E + 2] += wf * evw * f0;
    }
    const double Iw = m.sigma_R * Tw * Tw * Tw * Tw / PI;
    for (int o = threadIdx.x; o < oq.n; o += MF_NT) {
        double on = 0.0;
        for (int a = 0; a < DIM; ++a) on += oq.x[a * oq.n_pad + o] * n[a];
        if (on > 0.0) acc[NS] += oq.w[o] * on / (4.0 * PI);
        else acc[NS + 1] += oq.w[o] * on * Iw;
    }
    cta_sum<NS + 2>(acc, buf);
    if (threadIdx.x != 0) return;
    for (int k = 0; k < NS + 2; ++k) binc[(size_t)b * BINC + k] = acc[k];
    binc[(size_t)b * BINC + NS + 2] = 1.0 / acc[0];
}

// Blocks [0, n_face_cta): MF_FACES interior faces each; the first half of the threads
// evaluates the Rusanov flux of a face, the second half its NSF and high-order terms and its
// Gamma (two chains of similar length instead of one of twice it).  Fx [n_fi][NVM] is the
// flux times the area, owner -> neighbour; fgam [n_fi][2] the Gammas times the area.
// Blocks [n_face_cta, n_face_cta + n_bf): one boundary face each.  The rest: the sources of
// MF_NT cells each, src [nc][SRC].
template <typename R, int DIM, int ORDER>
__device__ __forceinline__ void k_macro_flux_body(MacroGeom g, ModelDev m, QuadD vq, int n_face_cta, int n_bf_cta, const MacroState *__restrict__ st, const R *__restrict__ grad, const R *__restrict__ rec, R *__restrict__ Fx, R *__restrict__ fgam, R *__restrict__ src, double *__restrict__ bflux) {
    constexpr int NV = DIM + 5, E = 1 + DIM;
    if (st && st->done) return;
    const MacroReal<R> &c = real<R>(g);
    if ((int)blockIdx.x < n_face_cta) {
        __shared__ R conv[E + 3][MF_FACES];
        const int l = threadIdx.x % MF_FACES, f = blockIdx.x * MF_FACES + l;
        const bool first = threadIdx.x < MF_FACES, valid = f < g.n_fi;
        const int4 fi = valid ? g.fi4[f] : make_int4(0, 0, 0, 0);
        const R *G = c.fgeo + (size_t)(valid ? f : 0) * FGEO;
        const R S = G[11];
        if (first && valid) {
            const R *qL = ORDER == 2 ? rec + ((size_t)fi.x * MAXF + fi.z) * NVM : c.q + (size_t)fi.x * NVM;
            const R *qR = ORDER == 2 ? rec + ((size_t)fi.y * MAXF + fi.w) * NVM : c.q + (size_t)fi.y * NVM;
            R n[DIM], F[NV];
#pragma unroll
            for (int a = 0; a < DIM; ++a) n[a] = G[a];
            rusanov<R, DIM>(qL, qR, n, S, m, c, F);
#pragma unroll
            for (int k = 0; k < E + 3; ++k) conv[k][l] = F[k];
        }
        R F[NV];
        if (!first && valid) {
            R pf[NV], mu, irho, kR, sn[DIM], qn[4];
            nsf_normal<R, DIM>(g, m, G, fi.x, fi.y, grad, pf, mu, irho, kR, sn, qn);
            const R idn = G[12];
            const R *h = c.hot + (size_t)f * NVM;
            R un = R(0), unf = R(0);
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                sn[a] += h[a];
                un = fma(sn[a], pf[1 + a], un);
                unf = fma(pf[1 + a], G[a], unf);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) qn[k] += h[DIM + k];
            F[0] = R(0);
#pragma unroll
            for (int a = 0; a < DIM; ++a) F[1 + a] = S * sn[a];
            F[E] = S * (un + ((qn[0] + qn[1]) + (qn[2] + qn[3])));
#pragma unroll
            for (int k = 1; k < 4; ++k) F[E + k] = S * qn[k];
            fgam[(size_t)f * 2] = S * (fabs(unf) + sound_speed(pf[E]) + R(2) * mu * irho * idn);
            fgam[(size_t)f * 2 + 1] = S * (R(2) * kR * idn);
        }
        __syncthreads();
        if (!first && valid) {
#pragma unroll
            for (int k = 0; k < NV; ++k) Fx[(size_t)f * NVM + k] = k < E + 3 ? F[k] + conv[k][l] : F[k];
        }
        return;
    }
    const int b = (int)blockIdx.x - n_face_cta;
    if (b < n_bf_cta) {
        boundary_face<R, DIM>(g, m, vq, b, bflux);
        return;
    }
    // sources Q of Section 5 (rotational and vibrational relaxation, gas-photon exchange) and
    // the nonzero entries of their Jacobian d(Q_egas, Q_r, Q_v, Q_R)/d(e_gas, e_r, e_v, e_R)
    // with rho, rho u, tau, k_eff frozen:
    //   [ 0, 0, -kb, k ], [ c, -cr, -c, 0 ], [ e, -e, -zv - kb, k ], [ 0, 0, kb, -k ]
    // c = d_r / (3 + d_r) zr, cr = zr, zr = 1 / (Z_r tau); e = 2 eps'(T_tv) / (3 + 2 eps'(T_tv)) zv,
    // zv = 1 / (Z_v tau); kb = k_eff 16 sigma_R T_v^3 / (rho eps'(T_v)), eps(T) = d_v(T) T / 2.
    const int i = (b - n_bf_cta) * MF_NT + threadIdx.x;
    if (i >= g.n_cells) return;
    const R *q = c.q + (size_t)i * NVM;
    const R rho = q[0], Tt = q[E], Tr = q[E + 1], Tv = q[E + 2], eR = q[E + 3];
    const R itau = rho * pow_r(Tt, R(1) - c.omega) * c.i_mu0;      // 1 / tau
    const R zr = itau * c.i_Zr, zv = itau * c.i_Zv, k = absorption(rho, c);
    const R s3 = R(4) * c.sigma * Tv * Tv * Tv, ex = k * fma(s3, Tv, -eR);
    R *o = src + (size_t)i * SRC;
    o[0] = c.half_dr * rho * c.w_r * (Tt - Tr) * zr;               // T_tr - T_r = 3 (T_t - T_r) / (3 + d_r)
    R cvv, ctv, dev;                                               // eps'(T_v), eps'(T_tv), eps(T_tv) - eps(T_v)
    if (m.dv_T) {
        const R ev = vib_energy<R>(m, Tv), Ttv = equal_temperature<R>(m, R(3), R(3) * Tt + R(2) * ev);
        cvv = vib_cv<R>(m, Tv);
        ctv = vib_cv<R>(m, Ttv);
        dev = vib_energy<R>(m, Ttv) - ev;
        o[8] = R(2) * ctv * rcp_r(fma(R(2), ctv, R(3))) * zv;
        o[4] = R(4) * k * s3 * rcp_r(rho * cvv);
    } else {
        dev = c.half_dv * c.w_v * (Tt - Tv);
        o[8] = c.e_v * zv;
        o[4] = R(4) * k * s3 * (c.i_half_dv * rcp_r(rho));
    }
    o[1] = fma(rho * dev, zv, -ex);
    o[2] = ex;
    R uu = R(0), ke = R(0);
#pragma unroll
    for (int a = 0; a < DIM; ++a) uu = fma(q[1 + a], q[1 + a], uu);
    o[3] = (sqrt_r(uu) + sound_speed(Tt)) * c.icdx[i];             // 1 / dt
    o[5] = k;
    o[6] = c.c_r * zr;
    o[7] = zr;
    o[9] = zv;
    // the state that the relaxation's flux increments need: H = E_gas + p, e_r, e_v
    const R p = rho * Tt, er = c.half_dr * rho * Tr, ev = rho * vib_e(Tv, m, c);
    ke = rho * uu;
    o[10] = fma(R(2.5), p, fma(R(0.5), ke, er + ev));
    o[11] = er;
    o[12] = ev;
}
template <typename R, int DIM, int ORDER>
__global__ void __launch_bounds__(MF_NT) k_macro_flux(MacroGeom g, ModelDev m, QuadD vq, int n_face_cta, int n_bf_cta, const MacroState *st, const R *grad, const R *rec, R *Fx, R *fgam, R *src, double *bflux) {
    wait_for_previous();
    k_macro_flux_body<R, DIM, ORDER>(g, m, vq, n_face_cta, n_bf_cta, st, grad, rec, Fx, fgam, src, bflux);
}

// ------------------------------------------------------------------ high-order terms
// one thread per interior face, then one per boundary face; hot [n_fi][NVM]: stress . n
// (DIM), then the four heat fluxes . n
template <typename R, int DIM>
__global__ void k_macro_hot(MacroGeom g, ModelDev m, const double *__restrict__ Fk, const R *__restrict__ grad,
                            const double *__restrict__ kin_bflux, const double *__restrict__ mac_bflux,
                            double *__restrict__ hot, float *__restrict__ hotf, double *__restrict__ hot_b) {
    constexpr int NV = DIM + 5;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < g.n_fi) {
        const MacroReal<R> &c = real<R>(g);
        const int4 fi = g.fi4[t];
        R pf[NV], mu, irho, kR, sn[DIM], qn[4];
        nsf_normal<R, DIM>(g, m, c.fgeo + (size_t)t * FGEO, fi.x, fi.y, grad, pf, mu, irho, kR, sn, qn);
        const double *n = g.d.fgeo + (size_t)t * FGEO;
        const double *ri = Fk + (size_t)fi.x * NF, *rj = Fk + (size_t)fi.y * NF;
        double *h = hot + (size_t)t * NVM;
        double x[DIM + 4];
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            x[a] = -to_double(sn[a]);
#pragma unroll
            for (int b = 0; b < DIM; ++b) {
                // record words of the stress: xx, yy, zz, xy, xz, yz at 20
                const int k = a == b ? 20 + a : 22 + a + b;
                x[a] = fma(0.5 * (ri[k] + rj[k]), n[b], x[a]);
            }
        }
#pragma unroll
        for (int md = 0; md < 4; ++md) {
            x[DIM + md] = -to_double(qn[md]);
#pragma unroll
            for (int d = 0; d < DIM; ++d) x[DIM + md] = fma(0.5 * (ri[8 + 3 * md + d] + rj[8 + 3 * md + d]), n[d], x[DIM + md]);
        }
#pragma unroll
        for (int k = 0; k < DIM + 4; ++k) {
            h[k] = x[k];
            if (hotf) hotf[(size_t)t * NVM + k] = fp64::narrow(x[k]);
        }
        return;
    }
    const int b = t - g.n_fi;
    if (b < g.n_bf)
        for (int k = 0; k < NV; ++k)
            hot_b[(size_t)b * NVM + k] = kin_bflux[(size_t)b * NVM + k] - mac_bflux[(size_t)b * NVM + k];
}

// ------------------------------------------------------------------ residual and relaxation
constexpr int DSTR = 24;       // Dinv record: NVM diagonal inverses (first E used), 4x4 block

namespace {

// D of the energy rows, diag(d0, d0, d0, dR) minus the source Jacobian above, eliminated
// photons first, then gas energy and e_r in terms of e_v.  Every pivot is a sum of positive
// terms: dR + k, d0, d0 + zr, and the last one, d0 + zv + kb dR/(dR + k) + e (g - h), with
// e < zv and h - g < c / (d0 + zr) < 1.
template <typename T>
struct EnergyD {
    T ir3, k, id0, i1, c, e, g, h, is, kbi;
    __device__ __forceinline__ EnergyD(T d0, T dR, T kb, T k_, T c_, T zr, T e_, T zv) {
        k = k_;
        c = c_;
        e = e_;
        ir3 = rcp_r(dR + k);
        id0 = rcp_r(d0);
        i1 = rcp_r(d0 + zr);
        kbi = kb * ir3;
        const T w = kbi * dR;
        g = w * id0;
        h = fma(c, g, c) * i1;
        is = rcp_r(fma(e, g - h, d0 + zv + w));
    }
    // the same elimination with its coefficients widened
    template <typename S>
    __device__ __forceinline__ explicit EnergyD(const EnergyD<S> &o)
        : ir3(to_double(o.ir3)), k(to_double(o.k)), id0(to_double(o.id0)), i1(to_double(o.i1)), c(to_double(o.c)),
          e(to_double(o.e)), g(to_double(o.g)), h(to_double(o.h)), is(to_double(o.is)), kbi(to_double(o.kbi)) {}
    __device__ __forceinline__ void solve(T b0, T b1, T b2, T b3, T (&x)[4]) const {
        const T t3 = b3 * ir3;
        const T y0 = fma(k, t3, b0) * id0, y1 = fma(c, y0, b1) * i1;
        x[2] = fma(e, y0 - y1, fma(k, t3, b2)) * is;
        x[0] = fma(-g, x[2], y0);
        x[1] = fma(-h, x[2], y1);
        x[3] = fma(kbi, x[2], t3);
    }
};

// Increment of the convective flux vectors, F_a(W + dW) - F_a(W) in every direction a,
// without forming either flux: every term is a product of an increment with a state value,
// so that its rounding is relative to the increment.
//   rho1 = rho + drho, du = (dm - u drho) / rho1, d(rho |u|^2) = drho |u1|^2 + rho du.(u1 + u),
//   dp = 2/3 (dEg - der - dev - d(rho |u|^2) / 2),
//   d(m_b u_a) = dm_b u_a1 + m_b du_a, d(u_a X) = du_a X1 + u_a dX (X = Eg + p, e_r, e_v).
template <typename R, int DIM>
struct FluxIncrement {
    R du[DIM], u1[DIM], dp, dH;
    __device__ __forceinline__ FluxIncrement(R rho, const R *u, R drho, const R *dm, R dEg, R der, R dev) {
        const R inv1 = rcp_r(rho + drho);
        R uu1 = R(0), dq = R(0);
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            du[a] = fma(-u[a], drho, dm[a]) * inv1;
            u1[a] = u[a] + du[a];
            uu1 = fma(u1[a], u1[a], uu1);
            dq = fma(du[a], u1[a] + u[a], dq);
        }
        dp = R(2.0 / 3.0) * fma(R(-0.5), fma(drho, uu1, rho * dq), dEg - der - dev);
        dH = dEg + dp;
    }
};

// One relaxation record per (cell, row): the flux increment vector of the row (DIM values)
// and the row's dW at [3] (FP64: 32 bytes, FP32: 16)
template <typename R>
struct __align__(4 * sizeof(R)) Row {
    R x[4];
};

}  // namespace

// Eight lanes per cell, lane v = row v.  The first relaxation sweep has no neighbour terms
// (dW = D^-1 R) and is made here.  With `st`, the last CTA to finish (an atomic ticket after
// a fence, no waiting) adds the CTA partials of |R|^2 in a fixed order and sets the norm,
// the iteration count and the stop flag.
template <typename R, int DIM>
__device__ __forceinline__ void k_macro_residual_body(MacroGeom g, MacroState *__restrict__ st, const R *__restrict__ Fx, const R *__restrict__ fgam, const R *__restrict__ src, const double *__restrict__ bflux, const double *__restrict__ hot_b, double *__restrict__ Rg, double *__restrict__ Dinv, R *__restrict__ gam, Row<R> *__restrict__ rows, double *__restrict__ rpart, double *__restrict__ history) {
    constexpr int NV = DIM + 5, E = 1 + DIM, ER = 4 + DIM;
    if (st && st->done) return;
    const MacroReal<R> &c = real<R>(g);
    const int t = blockIdx.x * blockDim.x + threadIdx.x, v = t % NVM;
    const bool valid = t / NVM < g.n_cells;
    const int i = valid ? t / NVM : g.n_cells - 1;
    const unsigned lane = threadIdx.x & 31;
    const int l0 = (int)(lane & ~(unsigned)(NVM - 1));       // the cell's first lane
    const int nf = g.info[i].x;
    const R *q = c.q + (size_t)i * NVM;
    const R hiv = c.hivol[i];
    R acc = R(0), gs = R(0), gsR = R(0);
#pragma unroll
    for (int k = 0; k < MAXF; ++k) {
        if (k >= nf) break;
        const int fid = g.cface[i * MAXF + k];
        if (fid >= 0) {
            if (v < NV) {
                const R x = Fx[(size_t)fid * NVM + v];
                acc = g.own[i * MAXF + k] ? acc - x : acc + x;
            }
            const R gb = fgam[(size_t)fid * 2], gR = fgam[(size_t)fid * 2 + 1];
            gs += gb;
            gsR += gR;
            if (v < 2 && valid) gam[((size_t)i * MAXF + k) * 2 + v] = v == 0 ? gb * hiv : (gb + gR) * hiv;
        } else {
            const int b = -1 - fid;
            const R *bg = c.bgeo + (size_t)b * 8;
            const R S = bg[3], idn = bg[4];
            if (v < NV) {
                const double x = bflux[(size_t)b * NVM + v] + hot_b[(size_t)b * NVM + v];
                acc = fma(-to_real<R>(x), S, acc);
            }
            R un = R(0);
#pragma unroll
            for (int a = 0; a < DIM; ++a) un = fma(q[1 + a], bg[a], un);
            const bool mirror = g.patch_kind[g.bf_patch[b]] == 2;
            // a mirror face: the Rusanov part only, and nothing in the e_R row
            R gb = fabs(un) + sound_speed(q[E]), gR = -gb;
            if (!mirror) {
                const R ir = rcp_r(q[0]);
                gb += R(2) * viscosity(q[E], c) * ir * idn;
                gR = R(2) * (c.dens ? c.kR0 * ir : c.kR0) * idn;
            }
            gs = fma(gb, S, gs);
            gsR = fma(gR, S, gsR);
        }
    }
    const R *so = src + (size_t)i * SRC;
    const R iv = c.ivol[i];
    R r = acc * iv;
    if (v > E && v < NV) r += so[v - E - 1];
    if (g.moff && v < NV) r += to_real<R>(g.moff[(size_t)i * NVM + v]);
    const double r8 = v < NV && valid ? to_double(r) : 0.0;
    double r2 = r8 * r8;
    // relaxation form: the energy row holds the gas energy
    const double rR = __shfl_sync(0xffffffffu, r8, l0 + ER);
    const double rg = v == E ? r8 - rR : r8;
    if (valid && v < NV) Rg[(size_t)i * NVM + v] = rg;
    const R d0 = fma(gs, iv, so[3]), dR = fma(gs + gsR, iv, so[3]);
    const EnergyD<R> D(d0, dR, so[4], so[5], so[6], so[7], so[8], so[9]);
    double *Di = Dinv + (size_t)i * DSTR;
    if (valid) {
        if (v == 0) Di[0] = to_double(D.id0);
        if (v < 4) {       // lane v: column v of the inverse
            R x[4];
            D.solve(R(v == 0), R(v == 1), R(v == 2), R(v == 3), x);
#pragma unroll
            for (int k = 0; k < 4; ++k) Di[NVM + k * 4 + v] = to_double(x[k]);
        }
    }
    // first sweep: dW = D^-1 R (in FP64), and its flux increments
    double rr[NV], x4[4];
#pragma unroll
    for (int k = 0; k < NV; ++k) rr[k] = __shfl_sync(0xffffffffu, rg, l0 + k);
    if constexpr (sizeof(R) == 8) {
        D.solve(rr[E], rr[E + 1], rr[E + 2], rr[E + 3], x4);
    } else {
        const EnergyD<double> D8(D);
        D8.solve(rr[E], rr[E + 1], rr[E + 2], rr[E + 3], x4);
    }
    const double id0 = to_double(D.id0);
    R u[DIM], dm[DIM];
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        u[a] = q[1 + a];
        dm[a] = to_real<R>(id0 * rr[1 + a]);
    }
    const R drho = to_real<R>(id0 * rr[0]), dEg = to_real<R>(x4[0]), der = to_real<R>(x4[1]),
            dev = to_real<R>(x4[2]), deR = to_real<R>(x4[3]);
    const FluxIncrement<R, DIM> fi(q[0], u, drho, dm, dEg, der, dev);
    if (valid && v < NV) {
        Row<R> o;
        o.x[1] = o.x[2] = R(0);
        if (v <= DIM) {
            R dmb = drho;
#pragma unroll
            for (int a = 0; a < DIM; ++a)
                if (v == 1 + a) dmb = dm[a];
            const R mb = v == 0 ? R(0) : q[0] * q[v];
#pragma unroll
            for (int a = 0; a < DIM; ++a)
                o.x[a] = v == 0 ? dm[a] : fma(dmb, fi.u1[a], fma(mb, fi.du[a], v == 1 + a ? fi.dp : R(0)));
            o.x[3] = dmb;
        } else {
            const R X = v == ER ? R(0) : so[10 + v - E], dX = v == E ? fi.dH : v == E + 1 ? der : v == E + 2 ? dev : R(0);
            const R X1 = X + dX;
#pragma unroll
            for (int a = 0; a < DIM; ++a) o.x[a] = fma(fi.du[a], X1, u[a] * dX);
            o.x[3] = v == E ? dEg : v == E + 1 ? der : v == E + 2 ? dev : deR;
        }
        rows[(size_t)i * NVM + v] = o;
    }
    if (!st) return;
    // deterministic per-CTA partial of |R|^2, then the last CTA
    __shared__ double ws[4];
    __shared__ bool last;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r2 += __shfl_xor_sync(0xffffffffu, r2, o);
    if (lane == 0) ws[threadIdx.x >> 5] = r2;
    __syncthreads();
    if (threadIdx.x == 0) {
        rpart[blockIdx.x] = (ws[0] + ws[1]) + (ws[2] + ws[3]);
        __threadfence();
        last = atomicAdd(&st->ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double s = 0.0;
    for (unsigned k = threadIdx.x; k < gridDim.x; k += blockDim.x) s += __ldcg(rpart + k);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) ws[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x != 0) return;
    st->ticket = 0u;
    if (st->it >= st->max_inner) {
        st->done = 1;
        return;
    }
    const double rn = sqrt((ws[0] + ws[1]) + (ws[2] + ws[3]));
    if (st->it == 0) st->r0 = rn;
    st->rn = rn;
    if (history) history[st->it] = rn;
    st->it += 1;
    if (!isfinite(rn) || rn <= st->tol * st->r0) st->done = 1;
}
template <typename R, int DIM>
__global__ void __launch_bounds__(128) k_macro_residual(MacroGeom g, MacroState *st, const R *Fx, const R *fgam, const R *src, const double *bflux, const double *hot_b, double *Rg, double *Dinv, R *gam, Row<R> *rows, double *rpart, double *history) {
    wait_for_previous();
    k_macro_residual_body<R, DIM>(g, st, Fx, fgam, src, bflux, hot_b, Rg, Dinv, gam, rows, rpart, history);
}

// One point-relaxation sweep from the neighbours' records of the previous sweep.  Four lanes
// per cell: lane r holds row r (r < E) and row r of the energy block, so that its two rows'
// neighbour terms, its row of the block's inverse and its two output rows are its own, and
// only the increments are exchanged (by shuffles).  R = double: everything in FP64;
// R = float: the neighbour terms in FP32 (as stored), their sum, the solve and the update in
// FP64.  FIRST: no neighbour terms.  LAST: W += dW and the primitive variables of the new W.
template <typename R, int DIM, bool FIRST, bool LAST>
__device__ __forceinline__ void k_macro_jacobi_body(MacroGeom g, ModelDev m, const MacroState *__restrict__ st, const double *__restrict__ Rg, const double *__restrict__ Dinv, const R *__restrict__ gam, const R *__restrict__ src, const Row<R> *__restrict__ in, Row<R> *__restrict__ out, double *__restrict__ W, double *__restrict__ qd, float *__restrict__ qf) {
    constexpr int E = 1 + DIM, LPC = 4;
    if (st->done) return;
    const MacroReal<R> &c = real<R>(g);
    const int t = blockIdx.x * blockDim.x + threadIdx.x, r = t % LPC;
    const bool valid = t / LPC < g.n_cells;
    const int i = valid ? t / LPC : g.n_cells - 1;
    const int l0 = (int)(threadIdx.x & 31 & ~(LPC - 1));
    const bool two = r < E;        // row r of the first block exists (E = 2, 3, 4)
    double x0 = two ? Rg[(size_t)i * NVM + r] : 0.0, x1 = Rg[(size_t)i * NVM + E + r];
    if constexpr (!FIRST) {
        const int4 nb = *reinterpret_cast<const int4 *>(g.nb + (size_t)i * MAXF);
        const int nbk[MAXF] = {nb.x, nb.y, nb.z, nb.w};
        Row<R> a0[MAXF], a1[MAXF];
#pragma unroll
        for (int k = 0; k < MAXF; ++k) {
            const size_t o = (size_t)max(nbk[k], 0) * NVM;
            if (nbk[k] >= 0) {
                a0[k] = in[o + (two ? r : 0)];
                a1[k] = in[o + E + r];
            }
        }
#pragma unroll
        for (int k = 0; k < MAXF; ++k) {
            if (nbk[k] < 0) continue;
            const R *nS = c.cnS + ((size_t)i * MAXF + k) * MGS;
            const R gb = gam[((size_t)i * MAXF + k) * 2], gE = r == 3 ? gam[((size_t)i * MAXF + k) * 2 + 1] : gb;
            if constexpr (sizeof(R) == 8) {
                x0 = fma(gb, a0[k].x[3], x0);
                x1 = fma(gE, a1[k].x[3], x1);
#pragma unroll
                for (int a = 0; a < DIM; ++a) {
                    x0 = fma(-nS[a], a0[k].x[a], x0);
                    x1 = fma(-nS[a], a1[k].x[a], x1);
                }
            } else {
                R t0 = -gb * a0[k].x[3], t1 = -gE * a1[k].x[3];
#pragma unroll
                for (int a = 0; a < DIM; ++a) {
                    t0 = fma(nS[a], a0[k].x[a], t0);
                    t1 = fma(nS[a], a1[k].x[a], t1);
                }
                x0 -= to_double(t0);
                x1 -= to_double(t1);
            }
        }
    }
    const double *Di = Dinv + (size_t)i * DSTR;
    const double d0 = Di[0] * x0;
    double d1 = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) d1 = fma(Di[NVM + r * 4 + k], __shfl_sync(0xffffffffu, x1, l0 + k), d1);
    if constexpr (LAST) {
        const double dE3 = __shfl_sync(0xffffffffu, d1, l0 + 3);
        double w0 = 0.0, w1 = 0.0;
        if (two) w0 = W[(size_t)i * NVM + r] + d0;
        w1 = W[(size_t)i * NVM + E + r] + d1;
        if (r == 0) w1 += dE3;
        double w[DIM + 5], q[DIM + 5];
#pragma unroll
        for (int k = 0; k < E; ++k) w[k] = __shfl_sync(0xffffffffu, w0, l0 + k);
#pragma unroll
        for (int k = 0; k < 4; ++k) w[E + k] = __shfl_sync(0xffffffffu, w1, l0 + k);
        primitive<DIM>(w, m, g.d, q);
        if (!valid) return;
        double q0 = 0.0, q1 = q[E];
#pragma unroll
        for (int k = 0; k < E; ++k)
            if (k == r) q0 = q[k];
#pragma unroll
        for (int k = 1; k < 4; ++k)
            if (k == r) q1 = q[E + k];
        if (two) {
            W[(size_t)i * NVM + r] = w0;
            qd[(size_t)i * NVM + r] = q0;
            if (qf) qf[(size_t)i * NVM + r] = fp64::narrow(q0);
        }
        W[(size_t)i * NVM + E + r] = w1;
        qd[(size_t)i * NVM + E + r] = q1;
        if (qf) qf[(size_t)i * NVM + E + r] = fp64::narrow(q1);
    } else {
        const R s0 = to_real<R>(d0), s1 = to_real<R>(d1);
        const R *q = c.q + (size_t)i * NVM;
        R u[DIM], dm[DIM];
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            u[a] = q[1 + a];
            dm[a] = __shfl_sync(0xffffffffu, s0, l0 + 1 + a);
        }
        const R drho = __shfl_sync(0xffffffffu, s0, l0), dEg = __shfl_sync(0xffffffffu, s1, l0),
                der = __shfl_sync(0xffffffffu, s1, l0 + 1), dev = __shfl_sync(0xffffffffu, s1, l0 + 2);
        const R rho = q[0];
        const FluxIncrement<R, DIM> fi(rho, u, drho, dm, dEg, der, dev);
        if (!valid) return;
        if (two) {
            Row<R> o;
            o.x[1] = o.x[2] = R(0);
            const R mb = r == 0 ? R(0) : rho * q[r];
#pragma unroll
            for (int a = 0; a < DIM; ++a)
                o.x[a] = r == 0 ? dm[a] : fma(s0, fi.u1[a], fma(mb, fi.du[a], r == 1 + a ? fi.dp : R(0)));
            o.x[3] = s0;
            out[(size_t)i * NVM + r] = o;
        }
        Row<R> o;
        o.x[1] = o.x[2] = R(0);
        const R X = r == 3 ? R(0) : src[(size_t)i * SRC + 10 + r], dX = r == 0 ? fi.dH : r == 3 ? R(0) : s1, X1 = X + dX;
#pragma unroll
        for (int a = 0; a < DIM; ++a) o.x[a] = fma(fi.du[a], X1, u[a] * dX);
        o.x[3] = s1;
        out[(size_t)i * NVM + E + r] = o;
    }
}
template <typename R, int DIM, bool FIRST, bool LAST>
__global__ void __launch_bounds__(128) k_macro_jacobi(MacroGeom g, ModelDev m, const MacroState *st, const double *Rg, const double *Dinv, const R *gam, const R *src, const Row<R> *in, Row<R> *out, double *W, double *qd, float *qf) {
    wait_for_previous();
    k_macro_jacobi_body<R, DIM, FIRST, LAST>(g, m, st, Rg, Dinv, gam, src, in, out, W, qd, qf);
}

__global__ void k_macro_start(MacroState value, MacroState *st) { *st = value; }

// closed domains: fac = (total mass of the reference fields) / (total mass of W), the factor
// that k_macro_fields_from_W scales W by; CTA partials in a fixed order, added by the last CTA
constexpr int MM_CTAS = 64;
__global__ void __launch_bounds__(256) k_macro_mass(int n_cells, const double *__restrict__ vol,
                                                    const double *__restrict__ F_ref, const double *__restrict__ W,
                                                    double *__restrict__ part, MacroState *__restrict__ st,
                                                    double *__restrict__ fac) {
    __shared__ double a[8], b[8];
    __shared__ bool last;
    double sa = 0.0, sb = 0.0;
    auto reduce = [&] {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            sa += __shfl_xor_sync(0xffffffffu, sa, o);
            sb += __shfl_xor_sync(0xffffffffu, sb, o);
        }
        __syncthreads();
        if ((threadIdx.x & 31) == 0) {
            a[threadIdx.x >> 5] = sa;
            b[threadIdx.x >> 5] = sb;
        }
        __syncthreads();
        sa = sb = 0.0;
        for (int w = 0; w < 8; ++w) {
            sa += a[w];
            sb += b[w];
        }
    };
    for (int i = blockIdx.x * 256 + threadIdx.x; i < n_cells; i += gridDim.x * 256) {
        sa = fma(F_ref[(size_t)i * NF], vol[i], sa);
        sb = fma(W[(size_t)i * NVM], vol[i], sb);
    }
    reduce();
    if (threadIdx.x == 0) {
        part[blockIdx.x * 2] = sa;
        part[blockIdx.x * 2 + 1] = sb;
        __threadfence();
        last = atomicAdd(&st->ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    sa = sb = 0.0;
    if (threadIdx.x < gridDim.x) {
        sa = __ldcg(part + threadIdx.x * 2);
        sb = __ldcg(part + threadIdx.x * 2 + 1);
    }
    reduce();
    if (threadIdx.x == 0) {
        *fac = sa / sb;
        st->ticket = 0u;
    }
}

// ------------------------------------------------------------------ launchers
// 1-D and 2-D (3-D meshes take macro3d.cu)
#define MACRO_DISPATCH(dim, ...)          \
    do {                                  \
        if ((dim) == 1) {                 \
            constexpr int DIM = 1;        \
            __VA_ARGS__;                  \
        } else {                          \
            constexpr int DIM = 2;        \
            __VA_ARGS__;                  \
        }                                 \
    } while (0)

#define MACRO_DISPATCH_R(fp32, ...)      \
    do {                                  \
        if (fp32) {                       \
            using R = float;              \
            __VA_ARGS__;                  \
        } else {                          \
            using R = double;             \
            __VA_ARGS__;                  \
        }                                 \
    } while (0)

static int ctas(long long threads, int nt) { return (int)((threads + nt - 1) / nt); }

int macro_rpart_count(int n_cells) { return std::max(ctas((long long)n_cells * NVM, 128), 2 * MM_CTAS); }

cudaError_t launch_macro_start(cudaStream_t s, const MacroState &value, MacroState *st) {
    k_macro_start<<<1, 1, 0, s>>>(value, st);
    return cudaGetLastError();
}

cudaError_t launch_macro_from_fields(cudaStream_t s, int dim, int n_cells, const ModelDev &m, const double *F,
                                     const MacroWork &w) {
    MACRO_DISPATCH(dim, (k_macro_from_fields<DIM><<<ctas(n_cells, 64), 64, 0, s>>>(n_cells, m, F, w.W, w.qd, w.qf)));
    return cudaGetLastError();
}

cudaError_t launch_macro_fields_from_W(cudaStream_t s, const MacroGeom &g, const ModelDev &m, const MacroWork &w,
                                       const double *F_ref, double *F) {
    if (F_ref) {
        k_macro_mass<<<MM_CTAS, 256, 0, s>>>(g.n_cells, g.vol, F_ref, w.W, w.rpart, w.state, w.fac);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    MACRO_DISPATCH(g.dim, (k_macro_fields_from_W<DIM><<<ctas(g.n_cells, 64), 64, 0, s>>>(
                              g.n_cells, m, g.d, w.W, F_ref ? w.fac : nullptr, F)));
    return cudaGetLastError();
}

cudaError_t launch_macro_grad(cudaStream_t s, const MacroGeom &g, int order, int fp32, const MacroState *st,
                              const MacroWork &w) {
    const int nb = ctas((long long)g.n_cells * NVM, 128);
    MACRO_DISPATCH_R(fp32, MACRO_DISPATCH(g.dim, {
        if (order == 2) launch_after(s, k_macro_grad<R, DIM, 2>, nb, 128, g, st, (R *)w.grad, (R *)w.rec);
        else launch_after(s, k_macro_grad<R, DIM, 1>, nb, 128, g, st, (R *)w.grad, (R *)w.rec);
    }));
    return cudaGetLastError();
}

cudaError_t launch_macro_flux(cudaStream_t s, const MacroGeom &g, int order, int fp32, const ModelDev &m,
                              const QuadD &vq, const MacroState *st, const MacroWork &w, bool boundary_only) {
    const int nf = boundary_only ? 0 : ctas(g.n_fi, MF_FACES), nc = boundary_only ? 0 : ctas(g.n_cells, MF_NT);
    const int n = nf + g.n_bf + nc;
    if (n == 0) return cudaSuccess;
    MACRO_DISPATCH_R(fp32, MACRO_DISPATCH(g.dim, {
        if (order == 2)
            launch_after(s, k_macro_flux<R, DIM, 2>, n, MF_NT, g, m, vq, nf, g.n_bf, st, (const R *)w.grad, (const R *)w.rec,
                                                        (R *)w.Fx, (R *)w.fgam, (R *)w.src, w.mbf);
        else
            launch_after(s, k_macro_flux<R, DIM, 1>, n, MF_NT, g, m, vq, nf, g.n_bf, st, (const R *)w.grad, (const R *)w.rec,
                                                        (R *)w.Fx, (R *)w.fgam, (R *)w.src, w.mbf);
    }));
    return cudaGetLastError();
}

cudaError_t launch_macro_binc(cudaStream_t s, const MacroGeom &g, const ModelDev &m, const QuadD &vq, const QuadD &oq,
                              double *binc) {
    if (g.n_bf == 0) return cudaSuccess;
    MACRO_DISPATCH(g.dim, (k_macro_binc<DIM><<<g.n_bf, MF_NT, 0, s>>>(g, m, vq, oq, binc)));
    return cudaGetLastError();
}

cudaError_t launch_macro_hot(cudaStream_t s, const MacroGeom &g, int fp32, const ModelDev &m, const double *F_kin,
                             const MacroWork &w, const double *kin_bflux, double *hot_b) {
    const int n = g.n_fi + g.n_bf;
    if (n == 0) return cudaSuccess;
    MACRO_DISPATCH_R(fp32, MACRO_DISPATCH(g.dim, (k_macro_hot<R, DIM><<<ctas(n, 32), 32, 0, s>>>(
                                                     g, m, F_kin, (const R *)w.grad, kin_bflux, w.mbf, w.hot, w.hotf,
                                                     hot_b))));
    return cudaGetLastError();
}

cudaError_t launch_macro_residual(cudaStream_t s, const MacroGeom &g, int fp32, MacroState *st, const MacroWork &w,
                                  const double *hot_b, double *history) {
    const int nb = ctas((long long)g.n_cells * NVM, 128);
    MACRO_DISPATCH_R(fp32, MACRO_DISPATCH(g.dim, (launch_after(s, k_macro_residual<R, DIM>, nb, 128, 
                                                     g, st, (const R *)w.Fx, (const R *)w.fgam, (const R *)w.src, w.mbf,
                                                     hot_b, w.Rg, w.Dinv, (R *)w.gam, (Row<R> *)w.rows[0], w.rpart,
                                                     history))));
    return cudaGetLastError();
}

cudaError_t launch_macro_jacobi(cudaStream_t s, const MacroGeom &g, int fp32, const ModelDev &m, const MacroState *st,
                                int sweep, bool last, const MacroWork &w) {
    const int nb = ctas((long long)g.n_cells * 4, 128);
    MACRO_DISPATCH_R(fp32, MACRO_DISPATCH(g.dim, {
        const R *gam = (const R *)w.gam;
        const R *src = (const R *)w.src;
        const Row<R> *in = (const Row<R> *)w.rows[(sweep + 1) & 1];
        Row<R> *out = (Row<R> *)w.rows[sweep & 1];
        if (sweep == 0)
            launch_after(s, k_macro_jacobi<R, DIM, true, true>, nb, 128, g, m, st, w.Rg, w.Dinv, gam, src, in, out, w.W, w.qd,
                                                                  w.qf);
        else if (last)
            launch_after(s, k_macro_jacobi<R, DIM, false, true>, nb, 128, g, m, st, w.Rg, w.Dinv, gam, src, in, out, w.W,
                                                                   w.qd, w.qf);
        else
            launch_after(s, k_macro_jacobi<R, DIM, false, false>, nb, 128, g, m, st, w.Rg, w.Dinv, gam, src, in, out, w.W,
                                                                    w.qd, w.qf);
    }));
    return cudaGetLastError();
}

// Defect correction: moff = (kinetic residual rows) - R(W_h), from the relaxation form Rg of
// R(W_h) (whose total-energy row holds the gas energy, R_E - R_eR).
__global__ void k_macro_offset(int n_cells, int nv, const double *__restrict__ Rg, const double *__restrict__ rows,
                               double *__restrict__ moff) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_cells) return;
    const int E = nv - 4, ER = nv - 1;
    const double *rg = Rg + (size_t)i * NVM;
    for (int v = 0; v < nv; ++v) {
        const double Rh = v == E ? rg[E] + rg[ER] : rg[v];
        moff[(size_t)i * NVM + v] = rows[(size_t)i * NVM + v] - Rh;
    }
}

cudaError_t launch_macro_offset(cudaStream_t s, int dim, int n_cells, const double *Rg, const double *rows,
                                double *moff) {
    k_macro_offset<<<(n_cells + 127) / 128, 128, 0, s>>>(n_cells, dim + 5, Rg, rows, moff);
    return cudaGetLastError();
}

}  // namespace gsis
