// Device kernels of the GSIS library.
//
//  coefficients   per-cell reference-distribution coefficients from the FP64 fields
//                 (Section 2.1; Eq. reference_distribution)
//  wall_density   density of diffusely re-emitted molecules at each wall face
//  slopes         Venkatakrishnan-limited least-squares slopes of every (cell, velocity)
//                 and the upwind second-order value of every (interior face, velocity)
//                 that they give, for the residual of Eq. (deltaflux_micro)
//  sweep_gas      implicit finite-volume kinetic step of Eq. (dis_micro) for the four
//                 gas planes: upwind (order 1) or limited linear (order 2) residual,
//                 then forward/backward Gauss-Seidel point relaxation inside a block of
//                 consecutive cells, then the velocity moments of the new distribution
//                 (Eq. getmoment)
//  sweep_photon   the same step for the gray intensity I_R
//  finish         FP64 macroscopic fields from the moment partials, and the convergence
//                 measure of Section 6 (per-cell terms and their deterministic sum)
//  equilibrium    multi-temperature local equilibrium of given fields
//  moments_only   velocity moments of the current distributions
//
// Gas moments are taken about a shift velocity u0 per moment tile of MT consecutive
// cells (the velocity field of the tile's first cell), so that one tile shares one
// polynomial basis.  In FP32 the contraction over velocities can run on the tensor cores
// (tc_moments.cuh): in the standalone and synchronisation passes, and in the sweep's
// epilogue when a relaxation block lies inside one tile.
#include <algorithm>
#include <cmath>
#include <cooperative_groups.h>
#include <cstdio>
#include <type_traits>

#include "fp64.cuh"
#include "gsis_impl.cuh"
#include "tc_moments.cuh"

namespace gsis {

// ------------------------------------------------------------------ small vector type
template <typename Real, int N>
struct __align__(sizeof(Real) * N) Vec {
    Real v[N];
};

template <typename Real, int N>
__device__ __forceinline__ Vec<Real, N> vload(const Real *p) {
    return *reinterpret_cast<const Vec<Real, N> *>(p);
}
template <typename Real, int N>
__device__ __forceinline__ void vstore(Real *p, const Vec<Real, N> &x) {
    *reinterpret_cast<Vec<Real, N> *>(p) = x;
}

__device__ __forceinline__ float fexp(float x) { return __expf(x); }
__device__ __forceinline__ float expm1_r(float x) { return expm1f(x); }
__device__ __forceinline__ double expm1_r(double x) { return expm1(x); }
__device__ __forceinline__ double fexp(double x) { return exp(x); }

// x^(-DIM/2) of the Maxwellian normalisation (2 pi T)^(-DIM/2), without a general pow.
template <int DIM, typename T>
__device__ __forceinline__ T pow_neg_half_dim(T x) {
    if constexpr (DIM == 2) return T(1) / x;
    else if constexpr (DIM == 1) return T(1) / sqrt(x);
    else return T(1) / (x * sqrt(x));
}

// ------------------------------------------------------------------ coefficients
template <typename Real, int DIM>
__global__ void k_coefficients(Geom<Real> g, ModelDev m, const double *__restrict__ F,
                               const double *__restrict__ cell_dx, Real *__restrict__ coef) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n_cells) return;
    // computed in the storage precision: the coefficients are stored as Real
    using CT = Real;
    // a / b: in FP64 with fewer instructions (fp64.cuh)
    auto over = [](CT a, CT b) {
        if constexpr (std::is_same<CT, double>::value) return fp64::div_d(a, b);
        else return a / b;
    };
    const double *M = F + (size_t)i * NF;
    const CT rho = to_real<CT>(M[0]), Tt = to_real<CT>(M[4]), Tr = to_real<CT>(M[5]), Tv = to_real<CT>(M[6]);
    const CT dr = (CT)m.d_r, dv = (CT)m.d_v;
    const CT Ttr = over(CT(3) * Tt + dr * Tr, CT(3) + dr);
    // T_tv of Section 2.1; with the temperature-dependent d_v solved in FP64
    const double Ttv8 = m.dv_T ? equal_temperature<double>(m, 3.0, 3.0 * M[4] + 2.0 * vib_energy<double>(m, M[6])) : 0.0;
    const CT Ttv = m.dv_T ? (CT)Ttv8 : over(CT(3) * Tt + dv * Tv, CT(3) + dv);
    // the mixed heat fluxes and the radiative sink are differences of nearly equal terms
    // near equilibrium: they stay FP64
    double q[3][3];  // [mode t,r,v][component]
    for (int a = 0; a < 3; ++a) {
        q[0][a] = M[8 + a];
        q[1][a] = M[11 + a];
        q[2][a] = M[14 + a];
    }
    double Mc[9];     // Mix, per cell at d_v(T_v) when d_v depends on T_v
    if (m.dv_T) {
        double Ac[9];
        relaxation_matrix_at(m, dv_at(m, M[6]), Ac);
        mix_from_A(m, Ac, Mc);
    } else {
        for (int k = 0; k < 9; ++k) Mc[k] = m.Mix[k];
    }
    // q_t, q_r, q_v and q0, q1, q2 in the storage type (components past DIM are not read)
    CT qc[3][3], qa[3][3];
    for (int r = 0; r < 3; ++r)
        for (int a = 0; a < 3; ++a) {
            qc[r][a] = a < DIM ? to_real<CT>(q[r][a]) : CT(0);
            qa[r][a] = a < DIM ? to_real<CT>(Mc[r * 3 + 0] * q[0][a] + Mc[r * 3 + 1] * q[1][a] + Mc[r * 3 + 2] * q[2][a])
                               : CT(0);
        }
    const CT alpha[3] = {(CT)(1.0 - m.i_Zr - m.i_Zv), (CT)m.i_Zr, (CT)m.i_Zv};
    const CT Ta[3] = {Tt, Ttr, Ttv};
    const CT k1[3] = {CT(0.5) * dr * Tr, CT(0.5) * dr * Ttr, CT(0.5) * dr * Tr};
    // d_v(T) T / 2 at T_v (translational and rotational parts) and at T_tv (vibrational part)
    const CT ev = m.dv_T ? (CT)vib_energy<double>(m, M[6]) : CT(0.5) * dv * Tv;
    const CT etv = m.dv_T ? (CT)vib_energy<double>(m, Ttv8) : CT(0.5) * dv * Ttv;
    const CT k2[3] = {ev, ev, etv};
    Real *C = coef + (size_t)i * cf::NC;
    for (int a = 0; a < 3; ++a) C[cf::U + a] = to_real<CT>(M[1 + a]);
    const CT two_pi = (CT)6.283185307179586;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        Real *Cc = C + cf::COMP + c * cf::CSZ;
        const CT T = Ta[c];
        CT A, B, s, irT;
        if constexpr (std::is_same<CT, double>::value) {
            // one reciprocal each of T and rho T
            const CT iT = rcp_r(T);
            irT = rcp_r(rho * T);
            B = CT(0.5) * iT;
            const CT i2 = iT * CT(0.15915494309189535);
            A = alpha[c] * rho * (DIM == 2 ? i2 : DIM == 1 ? sqrt_r(i2) : i2 * sqrt_r(i2));
            s = CT(2.0 / 15.0) * iT * irT;
            Cc[cf::S] = B * CT(-fp64::EXP_SCALE);
            Cc[cf::A2] = A * (CT(3 - DIM) * T);
        } else {
            A = alpha[c] * rho * pow_neg_half_dim<DIM>(two_pi * T);
            B = CT(0.5) / T;
            Cc[cf::S] = CT(-0.7213475204444817) / T;      // -B log2 e
            Cc[cf::A2] = A * (CT(3 - DIM) * T);
            s = CT(2) / (CT(15) * T * rho * T);
            irT = CT(1) / (rho * T);
        }
        Cc[cf::A] = A;
        Cc[cf::B] = B;
        Cc[cf::T] = T;
        for (int a = 0; a < 3; ++a) {
            Cc[cf::Q + a] = s * (c == 0 ? qc[0][a] : qa[0][a]);
            Cc[cf::R1 + a] = (c == 0 ? qc[1][a] : qa[1][a]) * irT;
            Cc[cf::R2 + a] = (c == 0 ? qc[2][a] : qa[2][a]) * irT;
        }
        Cc[cf::K1] = k1[c];
        Cc[cf::K2] = k2[c];
    }
    const CT tau_rho = (CT)(0.7978845608028654 * m.Kn) * pow_r(Tt, (CT)(m.omega - 1.0));   // sqrt(2/pi) Kn
    const CT tau = over(tau_rho, rho);
    const CT keff = m.k_eff_density_scaled ? over(rho, (CT)m.Kn_p) : (CT)m.i_Knp;
    const CT ux = C[cf::U], uy = C[cf::U + 1], uz = C[cf::U + 2];
    const CT umag = sqrt_r(ux * ux + uy * uy + uz * uz);
    const CT sR = (CT)m.sigma_R;
    const double Tv8 = M[6], TR8 = M[7];
    const double sink = 4.0 * m.sigma_R * (Tv8 * Tv8 * Tv8 * Tv8 - TR8 * TR8 * TR8 * TR8);
    C[cf::RATE] = over(CT(1), tau);
    C[cf::INV_DT] = over(umag + sqrt_r(over(CT(5) * Tt, CT(3))), to_real<CT>(m.cfl_meso * cell_dx[i]));
    C[cf::SINK] = over(-keff * to_real<CT>(sink), rho);
    C[cf::GR] = over(sR * Tv * Tv * Tv * Tv, (CT)3.141592653589793);
    C[cf::KEFF] = keff;
}

// ------------------------------------------------------------------ wall density
// One warp per boundary face; far-field records are constant and left untouched.
template <typename Real, int DIM>
__global__ void k_wall_density(Geom<Real> g, Quad<Real> vq, const double *__restrict__ patch_T,
                               const double *__restrict__ bf_inc, const int *__restrict__ patch_kind,
                               const Real *__restrict__ f, const double *__restrict__ wout,
                               Real *__restrict__ bcoef) {
    // one CTA of WDT threads per boundary face: the outgoing mass flux of the current f,
    // summed per thread, per warp and then over the warps in a fixed order; the incoming
    // flux of the unit-density wall Maxwellian is a per-face constant (bf_inc)
    constexpr int WDT = 128;
    __shared__ double part[WDT / 32];
    const int face = blockIdx.x;
    const int p = g.bf_patch[face];
    if (patch_kind[p] != 0) return;
    const int cell = g.bf_cell[face];
    if (wout) {
        // velocity-sharded context: the outgoing flux over every rank's velocities
        if (threadIdx.x == 0) {
            const double inc = bf_inc[face];
            const double rho_w = inc < 0.0 ? -wout[face] / inc : 0.0;
            bcoef[(size_t)face * bc::NB + bc::A] = (Real)(rho_w * pow_neg_half_dim<DIM>(6.283185307179586 * patch_T[p]));
        }
        return;
    }
    Real n[DIM];
    for (int a = 0; a < DIM; ++a) n[a] = g.bf_nrm[face * 3 + a];
    double out = 0.0;
#pragma unroll 4
    for (int v = threadIdx.x; v < vq.n_pad; v += WDT) {
        Real xn = Real(0);
        for (int a = 0; a < DIM; ++a) xn += vq.x[a * vq.n_pad + v] * n[a];
        if (xn > Real(0)) out += (double)(vq.w[v] * xn) * (double)f[((size_t)cell * vq.n_pad + v) * 4];
    }
    for (int o = 16; o > 0; o >>= 1) out += __shfl_xor_sync(0xffffffffu, out, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = out;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int w = 0; w < WDT / 32; ++w) tot += part[w];
        const double inc = bf_inc[face];
        const double rho_w = inc < 0.0 ? -tot / inc : 0.0;
        const double norm = pow_neg_half_dim<DIM>(6.283185307179586 * patch_T[p]);
        bcoef[(size_t)face * bc::NB + bc::A] = (Real)(rho_w * norm);
    }
}

// Outgoing mass flux sum_{xi.n > 0} w xi.n F0 of the context's velocities at every wall
// face (zero at other boundary faces): the partial of a velocity shard, summed over the
// ranks before the next wall density.  Same per-face reduction order as k_wall_density.
template <typename Real, int DIM>
__global__ void k_wall_outflux(Geom<Real> g, Quad<Real> vq, const int *__restrict__ patch_kind,
                               const Real *__restrict__ f, double *__restrict__ wout) {
    constexpr int WDT = 128;
    __shared__ double part[WDT / 32];
    const int face = blockIdx.x;
    const int p = g.bf_patch[face];
    if (patch_kind[p] != 0) {
        if (threadIdx.x == 0) wout[face] = 0.0;
        return;
    }
    const int cell = g.bf_cell[face];
    Real n[DIM];
    for (int a = 0; a < DIM; ++a) n[a] = g.bf_nrm[face * 3 + a];
    double out = 0.0;
    for (int v = threadIdx.x; v < vq.n_pad; v += WDT) {
        Real xn = Real(0);
        for (int a = 0; a < DIM; ++a) xn += vq.x[a * vq.n_pad + v] * n[a];
        if (xn > Real(0)) out += (double)(vq.w[v] * xn) * (double)f[((size_t)cell * vq.n_pad + v) * 4];
    }
    for (int o = 16; o > 0; o >>= 1) out += __shfl_xor_sync(0xffffffffu, out, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = out;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int w = 0; w < WDT / 32; ++w) tot += part[w];
        wout[face] = tot;
    }
}

// ------------------------------------------------------------------ sweep helpers
template <typename Real, int N>
struct V {
    Real x[N];
};

template <typename Real, int N>
__device__ __forceinline__ V<Real, N> ldv(const Real *base, size_t idx) {
    V<Real, N> r;
    if constexpr (N == 1) {
        r.x[0] = base[idx];
    } else {
        Vec<Real, N> t = vload<Real, N>(base + idx * N);
#pragma unroll
        for (int p = 0; p < N; ++p) r.x[p] = t.v[p];
    }
    return r;
}

// Per-plane arithmetic.  An even number of FP32 planes runs on the packed FP32x2 pipe,
// two planes per instruction; each component rounds exactly as the scalar operation.
template <typename Real, int N>
__device__ __forceinline__ void vfma(Real c, const V<Real, N> &x, V<Real, N> &acc) {   // acc += c x
    if constexpr (std::is_same<Real, float>::value && N % 2 == 0) {
        const float2 cc = make_float2(c, c);
#pragma unroll
        for (int p = 0; p < N; p += 2) {
            const float2 r = __ffma2_rn(cc, make_float2(x.x[p], x.x[p + 1]), make_float2(acc.x[p], acc.x[p + 1]));
            acc.x[p] = r.x;
            acc.x[p + 1] = r.y;
        }
    } else {
#pragma unroll
        for (int p = 0; p < N; ++p) acc.x[p] = fma(c, x.x[p], acc.x[p]);
    }
}
template <typename Real, int N>
__device__ __forceinline__ V<Real, N> vadd(const V<Real, N> &a, const V<Real, N> &b) {
    V<Real, N> r;
    if constexpr (std::is_same<Real, float>::value && N % 2 == 0) {
#pragma unroll
        for (int p = 0; p < N; p += 2) {
            const float2 t = __fadd2_rn(make_float2(a.x[p], a.x[p + 1]), make_float2(b.x[p], b.x[p + 1]));
            r.x[p] = t.x;
            r.x[p + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int p = 0; p < N; ++p) r.x[p] = a.x[p] + b.x[p];
    }
    return r;
}
template <typename Real, int N>
__device__ __forceinline__ V<Real, N> vsub(const V<Real, N> &a, const V<Real, N> &b) {   // a - b
    V<Real, N> r;
    if constexpr (std::is_same<Real, float>::value && N % 2 == 0) {
        // b (-1) + a: the product is exact, so the one rounding is that of a - b
        const float2 m1 = make_float2(-1.0f, -1.0f);
#pragma unroll
        for (int p = 0; p < N; p += 2) {
            const float2 t = __ffma2_rn(make_float2(b.x[p], b.x[p + 1]), m1, make_float2(a.x[p], a.x[p + 1]));
            r.x[p] = t.x;
            r.x[p + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int p = 0; p < N; ++p) r.x[p] = a.x[p] - b.x[p];
    }
    return r;
}
template <typename Real, int N>
__device__ __forceinline__ V<Real, N> vmul(const V<Real, N> &a, const V<Real, N> &b) {
    V<Real, N> r;
    if constexpr (std::is_same<Real, float>::value && N % 2 == 0) {
#pragma unroll
        for (int p = 0; p < N; p += 2) {
            const float2 t = __fmul2_rn(make_float2(a.x[p], a.x[p + 1]), make_float2(b.x[p], b.x[p + 1]));
            r.x[p] = t.x;
            r.x[p + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int p = 0; p < N; ++p) r.x[p] = a.x[p] * b.x[p];
    }
    return r;
}
template <typename Real, int N>
__device__ __forceinline__ V<Real, N> vfmav(const V<Real, N> &a, const V<Real, N> &b, const V<Real, N> &c) {
    V<Real, N> r;   // a b + c per plane
    if constexpr (std::is_same<Real, float>::value && N % 2 == 0) {
#pragma unroll
        for (int p = 0; p < N; p += 2) {
            const float2 t = __ffma2_rn(make_float2(a.x[p], a.x[p + 1]), make_float2(b.x[p], b.x[p + 1]),
                                        make_float2(c.x[p], c.x[p + 1]));
            r.x[p] = t.x;
            r.x[p + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int p = 0; p < N; ++p) r.x[p] = fma(a.x[p], b.x[p], c.x[p]);
    }
    return r;
}
template <typename Real, int N>
__device__ __forceinline__ V<Real, N> vsplat(Real c) {
    V<Real, N> r;
#pragma unroll
    for (int p = 0; p < N; ++p) r.x[p] = c;
    return r;
}

// An int carried bit for bit in a Real slot (a face's upwind source, a stencil entry's cell).
__device__ __forceinline__ float int_bits_as(int x, float) { return __int_as_float(x); }
__device__ __forceinline__ double int_bits_as(int x, double) { return __longlong_as_double((long long)x); }
__device__ __forceinline__ int bits_as_int(float x) { return __float_as_int(x); }
__device__ __forceinline__ int bits_as_int(double x) { return (int)__double_as_longlong(x); }
template <typename Real>
struct Face {
    Real n[3], sv, svn, df[3], dn[3];
};

// The record of face k of cell c (layouts in gsis_impl.cuh: 8 Reals in 1-D/2-D, 12 in 3-D).
template <typename Real, int DIM = 2>
__device__ __forceinline__ Face<Real> load_face(const Real *__restrict__ fgeo, int c, int k) {
    const Real *p = fgeo + ((size_t)c * MAXF + k) * Lay<DIM>::FRS;
    const Vec<Real, 4> a = vload<Real, 4>(p), b = vload<Real, 4>(p + 4);
    Face<Real> F;
    if constexpr (DIM < 3) {
        F.n[0] = a.v[0];
        F.n[1] = a.v[1];
        F.sv = a.v[2];
        F.svn = a.v[3];
        F.df[0] = b.v[0];
        F.df[1] = b.v[1];
        F.dn[0] = b.v[2];
        F.dn[1] = b.v[3];
        F.n[2] = F.df[2] = F.dn[2] = Real(0);
    } else {
        const Vec<Real, 4> c3 = vload<Real, 4>(p + 8);
        F.n[0] = a.v[0];
        F.n[1] = a.v[1];
        F.n[2] = a.v[2];
        F.sv = a.v[3];
        F.svn = b.v[0];
        F.df[0] = b.v[1];
        F.df[1] = b.v[2];
        F.df[2] = b.v[3];
        F.dn[0] = c3.v[0];
        F.dn[1] = c3.v[1];
        F.dn[2] = c3.v[2];
    }
    return F;
}

// Reference distribution of the four gas planes at one (cell, velocity).
template <typename Real, int DIM>
__device__ __forceinline__ void reference(const Real *__restrict__ C, const Real *xi, Real (&gp)[4]) {
    constexpr int MH = 3 - DIM;
    const Vec<Real, 4> u4 = vload<Real, 4>(C + cf::U);
    Real c[DIM], c2 = Real(0);
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        c[a] = xi[a] - u4.v[a];
        c2 = fma(c[a], c[a], c2);
    }
    gp[0] = gp[1] = gp[2] = gp[3] = Real(0);
    if constexpr (std::is_same<Real, double>::value) {
        // 26 FP64 instructions per Maxwellian in 2-D (42 in the form below): the exponential's
        // scaled argument and A m T come with the coefficients, B T = 1/2 is used, and the
        // second bracket is the first plus q.c
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double *Ck = C + cf::COMP + k * cf::CSZ;
            const Vec<double, 4> a0 = vload<double, 4>(Ck), a1 = vload<double, 4>(Ck + 4), a2 = vload<double, 4>(Ck + 8),
                                 a3 = vload<double, 4>(Ck + 12);
            const double e = fp64::exp2n(a2.v[3], c2), E = a0.v[0] * e;
            double qc = a1.v[0] * c[0], r1 = a2.v[0] * c[0], r2 = a3.v[0] * c[0];
#pragma unroll
            for (int a = 1; a < DIM; ++a) {
                qc = fma(a1.v[a], c[a], qc);
                r1 = fma(a2.v[a], c[a], r1);
                r2 = fma(a3.v[a], c[a], r2);
            }
            const double p0 = fma(qc, fma(a0.v[1], c2, 0.5 * MH - 2.5), 1.0);
            gp[0] = fma(E, p0, gp[0]);
            if constexpr (MH > 0) gp[1] = fma(a3.v[3] * e, p0 + qc, gp[1]);
            gp[2] = fma(E, fma(a0.v[3], p0, r1), gp[2]);
            gp[3] = fma(E, fma(a1.v[3], p0, r2), gp[3]);
        }
        return;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const Real *Ck = C + cf::COMP + k * cf::CSZ;
        const Vec<Real, 4> a0 = vload<Real, 4>(Ck), a1 = vload<Real, 4>(Ck + 4), a2 = vload<Real, 4>(Ck + 8),
                           a3 = vload<Real, 4>(Ck + 12);
        const Real A = a0.v[0], Bk = a0.v[1], T = a0.v[2], K1 = a0.v[3], K2 = a1.v[3];
        const Real E = A * fexp(-Bk * c2);
        Real qc = Real(0), r1 = Real(0), r2 = Real(0);
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            qc = fma(a1.v[a], c[a], qc);
            r1 = fma(a2.v[a], c[a], r1);
            r2 = fma(a3.v[a], c[a], r2);
        }
        const Real p0 = fma(qc, fma(c2 + Real(MH) * T, Bk, Real(-2.5)), Real(1));
        gp[0] = fma(E, p0, gp[0]);
        if constexpr (MH > 0) {
            const Real ph = fma(qc, fma(c2 + Real(MH + 2) * T, Bk, Real(-2.5)), Real(1));
            gp[1] = fma(E * (Real(MH) * T), ph, gp[1]);
        }
        gp[2] = fma(E, fma(K1, p0, r1), gp[2]);
        gp[3] = fma(E, fma(K2, p0, r2), gp[3]);
    }
}

// Number of moments per gas chunk partial: F0: 1, c (DIM), cc (DIM(DIM+1)/2), c|c|^2 (DIM);
// H0 (DIM < 3): 1, c; f1: 1, c; f2: 1, c.
template <int DIM>
constexpr int n_gas_moments() {
    return 1 + DIM + DIM * (DIM + 1) / 2 + DIM + (DIM < 3 ? 3 : 2) * (1 + DIM);
}

// Accumulate the moments of one (cell, velocity) value into acc (shifted basis c = xi - u).
template <typename Real, int DIM>
__device__ __forceinline__ void add_moments(Real (&acc)[Lay<DIM>::NMP], const Real *c, Real w, const Real (&fv)[4]) {
    Real c2 = Real(0);
#pragma unroll
    for (int a = 0; a < DIM; ++a) c2 = fma(c[a], c[a], c2);
    const Real w0 = w * fv[0];
    int m = 0;
    acc[m++] += w0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) acc[m++] += w0 * c[a];
#pragma unroll
    for (int a = 0; a < DIM; ++a)
#pragma unroll
        for (int b = a; b < DIM; ++b) acc[m++] += w0 * c[a] * c[b];
#pragma unroll
    for (int a = 0; a < DIM; ++a) acc[m++] += w0 * c[a] * c2;
#pragma unroll
    for (int p = (DIM < 3 ? 1 : 2); p < 4; ++p) {
        const Real wp = w * fv[p];
        acc[m++] += wp;
#pragma unroll
        for (int a = 0; a < DIM; ++a) acc[m++] += wp * c[a];
    }
}

// ------------------------------------------------------------------ upwind face values
// Thread (tx, ty) of a 32 x SLOPE_ROWS CTA: cell blockIdx.x * SLOPE_ROWS + ty.  Computes the
// cell's least-squares gradient grad = sum_s C_js (f_s - f_j) over its stencil (face
// neighbours and their face neighbours), Venkatakrishnan's limiter phi = min(1, min_faces
// phi_V(Delta_1, Delta_2)) per plane, with the bounds Delta_1 taken over the interior face
// neighbours (the first entries of the stencil), and, on every interior face through which
// the velocity leaves the cell (xi . n > 0), the second-order reconstruction
// f_j + phi grad . (x_f - x_j) of every plane: fface[(face * n_pad + v) * N + plane].  The two
// cells of a face hold exactly opposite normals, so for each velocity exactly one of them (the
// upwind one) writes the face's value, and none where xi . n = 0, which the sweep skips.  The
// sweep reads these values for both its outflow and its inflow interior faces.
constexpr int SLOPE_ROWS = 8;
// velocities per thread of the FP32 pass (v, v + 32, ...), which share the cell's stencil
// indices, weights and face offsets
__host__ __device__ constexpr int slope_vpt(int dim) { return dim < 3 ? 2 : 1; }

// Row `i` of an array whose rows are `bytes` long: one 32 x 32 -> 64-bit multiply-add
__device__ __forceinline__ const float *row_at(const float *p, int i, unsigned bytes) {
    return reinterpret_cast<const float *>(reinterpret_cast<const char *>(p) + (unsigned long long)(unsigned)i * bytes);
}

// 1 / x to one unit in the last place, for normal x
__device__ __forceinline__ float rcp_normal(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// The FP32 slope pass.  It keeps the L1 data path (64 % of its cycles) and the issue slots
// (52 %) busier than memory (2.5 TB/s): per warp and pair of velocities 22 16-byte reads of f
// and some 60 broadcast reads of indices, weights and face records, each of which writes 32
// registers like any other (the weights as ready-made pairs cost more than the moves that
// make them: 313 us for what takes 254).  64 registers, four CTAs per SM: with Delta_2 of every
// face kept from the limiter to the reconstruction the pass runs three and takes 269 us.
// A row's address is one multiply-add, the two quotients of phi one reciprocal each, and the
// face loops have the cells' face count.  About 330 instructions per velocity, 501 before:
// 20 000 triangles x 784 velocities 324 -> 254 us, 40 000 x 2 304 1.89 -> 1.51 ms, 10 185
// tetrahedra x 4 096 1.31 -> 1.06 ms.
template <int N, int DIM, int FM>
__global__ void __launch_bounds__(32 * SLOPE_ROWS, 4) k_slopes32(Geom<float> g, int n, int n_pad,
                                                                                const float *__restrict__ xq,
                                                                                const float *__restrict__ f,
                                                                                float *__restrict__ fface) {
    // In 3-D the H0 plane carries nothing (no hidden velocity components): its gradient is
    // zero and no moment reads it, so its bounds and limiter are skipped (phi = 1).
    constexpr bool ZH = DIM == 3 && N == 4;
    constexpr int VPT = slope_vpt(DIM), MS = Lay<DIM>::MAXS, LW = Lay<DIM>::LW, FRS = Lay<DIM>::FRS;
    // stencil entries per batch, whose index and value loads are all issued before the batch
    // is used.  Entries past the stencil's end hold cell 0 and zero weights and add nothing.
    constexpr int BT = DIM < 3 ? 2 : 4;
    static_assert(MS % BT == 0, "batches tile the stencil records");
    const int v = blockIdx.y * (32 * VPT) + threadIdx.x;
    const int j = blockIdx.x * SLOPE_ROWS + threadIdx.y;
    if (j >= g.n_cells || blockIdx.y * (32 * VPT) >= n) return;   // no face value of a padding velocity is used
    const float *fv = f + (size_t)v * N;
    const unsigned row = (unsigned)n_pad * (N * 4);
    const int4 info = g.info[j];
    const int ns = info.y, nfn = info.z;
    V<float, N> fj[VPT], grad[VPT][DIM], dmax[VPT], dmin[VPT];
#pragma unroll
    for (int u = 0; u < VPT; ++u) {
        fj[u] = ldv<float, N>(row_at(fv, j, row), 32 * u);
        dmax[u] = dmin[u] = vsplat<float, N>(0.0f);
#pragma unroll
        for (int d = 0; d < DIM; ++d) grad[u][d] = vsplat<float, N>(0.0f);
    }
    const int *stn = g.stn + (size_t)j * MS;
    const float *lw = g.lsq + (size_t)j * MS * LW;
#pragma unroll
    for (int k0 = 0; k0 < MS; k0 += BT) {
        if (k0 >= ns) break;
        V<float, N> fs[BT][VPT];
#pragma unroll
        for (int t = 0; t < BT; ++t) {
            const float *p = row_at(fv, stn[k0 + t], row);
#pragma unroll
            for (int u = 0; u < VPT; ++u) fs[t][u] = ldv<float, N>(p, 32 * u);
        }
#pragma unroll
        for (int t = 0; t < BT; ++t) {
            const int k = k0 + t;
            float w[DIM];
#pragma unroll
            for (int d = 0; d < DIM; ++d) w[d] = lw[LW * k + d];
            const bool face_nbr = k < FM && k < nfn;
#pragma unroll
            for (int u = 0; u < VPT; ++u) {
                const V<float, N> dq = vsub(fs[t][u], fj[u]);
                if (face_nbr) {
#pragma unroll
                    for (int p = 0; p < N; ++p) {
                        if (ZH && p == 1) continue;
                        dmax[u].x[p] = fmaxf(dmax[u].x[p], dq.x[p]);
                        dmin[u].x[p] = fminf(dmin[u].x[p], dq.x[p]);
                    }
                }
#pragma unroll
                for (int d = 0; d < DIM; ++d) vfma(w[d], dq, grad[u][d]);
            }
        }
    }
    int fid[FM];             // < 0: boundary, or past the cell's faces
    float dx[FM][DIM];       // face centroid - cell centroid (zero where there is no interior face)
    const float *fg = g.fgeo + (size_t)j * MAXF * FRS;
#pragma unroll
    for (int k = 0; k < FM; ++k) {
        fid[k] = g.cface[(size_t)j * MAXF + k];
#pragma unroll
        for (int d = 0; d < DIM; ++d) dx[k][d] = fid[k] >= 0 ? fg[k * FRS + (DIM < 3 ? 4 : 5) + d] : 0.0f;
    }
    // Delta_2 = grad . (x_f - x_j) at the interior faces.  On the faces with Delta_2 > 0
    // (Delta_1 = Delta_max >= 0) phi_V >= 1 while Delta_2 <= Delta_1 / 2 and phi_V decreases for
    // Delta_2 > Delta_1 / 4, so the minimum is taken at the largest Delta_2; likewise at the most
    // negative Delta_2 with Delta_min.  Two evaluations per plane replace one per face.
    //   phi_V(d1, e) = num / den, num = d1 (d1 + 2 e) + eps2, den = d1 (d1 + e) + 2 e^2 + eps2
    //                = num + e (2 e - d1), which cancels at most a third of num.
    // den is at least eps2, kept a normal number (below it the squares of d1 and e vanish in
    // FP32 as well).
    const float eps2 = fmaxf(g.eps2[j], 1e-37f);
#pragma unroll
    for (int u = 0; u < VPT; ++u) {
        V<float, N> hi = vsplat<float, N>(0.0f), lo = hi;
#pragma unroll
        for (int k = 0; k < FM; ++k) {
            V<float, N> d2 = vmul(grad[u][0], vsplat<float, N>(dx[k][0]));
#pragma unroll
            for (int d = 1; d < DIM; ++d) vfma(dx[k][d], grad[u][d], d2);
#pragma unroll
            for (int p = 0; p < N; ++p) {
                if (ZH && p == 1) continue;
                hi.x[p] = fmaxf(hi.x[p], d2.x[p]);
                lo.x[p] = fminf(lo.x[p], d2.x[p]);
            }
        }
        const V<float, N> two = vsplat<float, N>(2.0f), ev = vsplat<float, N>(eps2);
        auto venkat = [&](const V<float, N> &d1, const V<float, N> &e) {
            const V<float, N> num = vfmav(d1, vfmav(two, e, d1), ev);
            const V<float, N> den = vfmav(e, vsub(vadd(e, e), d1), num);
            V<float, N> r;
#pragma unroll
            for (int p = 0; p < N; ++p) r.x[p] = (ZH && p == 1) ? 1.0f : num.x[p] * rcp_normal(den.x[p]);
            return r;
        };
        const V<float, N> ph = venkat(dmax[u], hi), pl = venkat(dmin[u], lo);
        V<float, N> phi;
#pragma unroll
        for (int p = 0; p < N; ++p) phi.x[p] = fminf(fminf(1.0f, ph.x[p]), pl.x[p]);
#pragma unroll
        for (int d = 0; d < DIM; ++d) grad[u][d] = vmul(grad[u][d], phi);
    }
#pragma unroll
    for (int k = 0; k < FM; ++k) {
        if (fid[k] < 0) continue;
        float nx[DIM];
#pragma unroll
        for (int d = 0; d < DIM; ++d) nx[d] = fg[k * FRS + d];
        float *o = const_cast<float *>(row_at(fface + (size_t)v * N, fid[k], row));
#pragma unroll
        for (int u = 0; u < VPT; ++u) {
            float xn = xq[v + 32 * u] * nx[0];
#pragma unroll
            for (int a = 1; a < DIM; ++a) xn = fmaf(xq[a * n_pad + v + 32 * u], nx[a], xn);
            V<float, N> val = fj[u];
#pragma unroll
            for (int d = 0; d < DIM; ++d) vfma(dx[k][d], grad[u][d], val);
            if (xn > 0.0f) {
                if constexpr (N == 1) {
                    o[32 * u] = val.x[0];
                } else {
                    Vec<float, N> t;
#pragma unroll
                    for (int p = 0; p < N; ++p) t.v[p] = val.x[p];
                    vstore<float, N>(o + 32 * u * N, t);
                }
            }
        }
    }
}

// The FP64 slope pass, one velocity per thread.  Its time is its FP64 instructions (19
// cycles of an SM each): the bounds and extremes are kept by integer comparisons of the bit
// patterns, every face's Delta_2 = grad . (x_f - x_j) is formed once and serves the limiter
// and the reconstruction f_j + phi Delta_2, and each plane takes one reciprocal: the smaller
// of the two quotients num / den of phi is found by cross-multiplication (all four terms
// are positive).  About 220 instructions per update in 2-D, 370 before (divisions 9 each,
// comparisons 1 to 2).  20 000 triangles x 784 velocities, order 2: 11.1 -> 5.9 ms.
template <int N, int DIM>
__global__ void __launch_bounds__(32 * SLOPE_ROWS) k_slopes64(Geom<double> g, int n, int n_pad,
                                                              const double *__restrict__ xq,
                                                              const double *__restrict__ f,
                                                              double *__restrict__ fface) {
    constexpr bool ZH = DIM == 3 && N == 4;      // the H0 plane of 3-D: slope not limited (phi = 1)
    constexpr int MS = Lay<DIM>::MAXS, LW = Lay<DIM>::LW;
    const int v = blockIdx.y * 32 + threadIdx.x;
    const int j = blockIdx.x * blockDim.y + threadIdx.y;
    if (j >= g.n_cells || blockIdx.y * 32 >= n) return;     // no face value of a padding velocity is used
    const V<double, N> fj = ldv<double, N>(f, (size_t)j * n_pad + v);
    const int4 info = g.info[j];
    const int *stn = g.stn + (size_t)j * MS;
    const double *lw = g.lsq + (size_t)j * MS * LW;
    double grad[DIM][N], dmax[N], dmin[N];
#pragma unroll
    for (int p = 0; p < N; ++p) {
        dmax[p] = 0.0;
        dmin[p] = -0.0;
#pragma unroll
        for (int d = 0; d < DIM; ++d) grad[d][p] = 0.0;
    }
#pragma unroll 2
    for (int k = 0; k < info.y; ++k) {
        const V<double, N> fs = ldv<double, N>(f, (size_t)stn[k] * n_pad + v);
        double c[DIM];
#pragma unroll
        for (int d = 0; d < DIM; ++d) c[d] = lw[LW * k + d];
#pragma unroll
        for (int p = 0; p < N; ++p) {
            const double dq = fs.x[p] - fj.x[p];
            if (k < info.z) {
                dmax[p] = max_pos(dmax[p], dq);
                dmin[p] = min_neg(dmin[p], dq);
            }
#pragma unroll
            for (int d = 0; d < DIM; ++d) grad[d][p] = fma(c[d], dq, grad[d][p]);
        }
    }
    // Delta_2 at the interior faces and their extremes
    double d2[MAXF][N], hi[N], lo[N];
    int fid[MAXF];
#pragma unroll
    for (int p = 0; p < N; ++p) {
        hi[p] = 0.0;
        lo[p] = -0.0;
    }
#pragma unroll
    for (int k = 0; k < MAXF; ++k) {
        fid[k] = k < info.x ? g.cface[j * MAXF + k] : -1;
        if (fid[k] < 0) continue;
        const double *q = g.fgeo + ((size_t)j * MAXF + k) * Lay<DIM>::FRS + (DIM < 3 ? 4 : 5);
#pragma unroll
        for (int p = 0; p < N; ++p) {
            d2[k][p] = grad[0][p] * q[0];
#pragma unroll
            for (int d = 1; d < DIM; ++d) d2[k][p] = fma(grad[d][p], q[d], d2[k][p]);
            hi[p] = max_pos(hi[p], d2[k][p]);
            lo[p] = min_neg(lo[p], d2[k][p]);
        }
    }
    const double eps2 = g.eps2[j];
    double phi[N];
#pragma unroll
    for (int p = 0; p < N; ++p) {
        phi[p] = 1.0;
        if (ZH && p == 1) continue;
        // phi_V(d1, d2) = num / den = (d1 (d1 + 2 d2) + eps2) / (d1 (d1 + d2) + 2 d2^2 + eps2)
        auto venkat = [&](double d1, double e, double &num, double &den) {
            const double t = d1 + e;
            num = fma(d1, t + e, eps2);
            den = fma(d1, t, fma(e + e, e, eps2));
        };
        double nh, dh, nl, dl;
        venkat(dmax[p], hi[p], nh, dh);
        venkat(dmin[p], lo[p], nl, dl);
        // positive numbers compare as their bit patterns
        const bool low = __double_as_longlong(nl * dh) < __double_as_longlong(nh * dl);
        const double num = low ? nl : nh, den = low ? dl : dh;
        if (__double_as_longlong(num) < __double_as_longlong(den)) phi[p] = num * fp64::rcp_d(den);
    }
    double xi[DIM];
#pragma unroll
    for (int a = 0; a < DIM; ++a) xi[a] = xq[a * n_pad + v];
#pragma unroll
    for (int k = 0; k < MAXF; ++k) {
        if (fid[k] < 0) continue;
        const Face<double> F = load_face<double, DIM>(g.fgeo, j, k);
        double xn = xi[0] * F.n[0];
#pragma unroll
        for (int a = 1; a < DIM; ++a) xn = fma(xi[a], F.n[a], xn);
        if (is_neg(xn) || is_zero(xn)) continue;
        Vec<double, N> t;
#pragma unroll
        for (int p = 0; p < N; ++p) t.v[p] = fma(phi[p], d2[k][p], fj.x[p]);
        vstore<double, N>(fface + ((size_t)fid[k] * n_pad + v) * N, t);
    }
}

__device__ __forceinline__ float neg_part(float a) { return fmin(a, 0.0f); }
__device__ __forceinline__ double neg_part(double a) { return is_neg(a) ? a : 0.0; }

// Sums of 24 values over eight consecutive lanes (sub = lane % 8, all lanes of the warp's
// group active): at each of three steps a lane passes one half of its values to its partner
// and adds the other half's; it ends with the sums of three values, x[q] holding number
// fold8_index(sub, q).
template <typename R>
__device__ __forceinline__ void fold8(R (&x)[24], int sub) {
    const unsigned mask = 0xFFu << ((threadIdx.x + blockDim.x * threadIdx.y) & 24u);
    const bool b2 = sub & 4, b1 = sub & 2, b0 = sub & 1;
#pragma unroll
    for (int m = 0; m < 12; ++m) {
        const R send = b2 ? x[m] : x[12 + m], keep = b2 ? x[12 + m] : x[m];
        x[m] = keep + __shfl_xor_sync(mask, send, 4);
    }
#pragma unroll
    for (int m = 0; m < 6; ++m) {
        const R send = b1 ? x[m] : x[6 + m], keep = b1 ? x[6 + m] : x[m];
        x[m] = keep + __shfl_xor_sync(mask, send, 2);
    }
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        const R send = b0 ? x[m] : x[3 + m], keep = b0 ? x[3 + m] : x[m];
        x[m] = keep + __shfl_xor_sync(mask, send, 1);
    }
}
__device__ __forceinline__ int fold8_index(int sub, int q) {
    return (sub & 4 ? 12 : 0) + (sub & 2 ? 6 : 0) + (sub & 1 ? 3 : 0) + q;
}

// ------------------------------------------------------------------ the sweep
// Shared memory of a sweep CTA: the main area (residuals and diagonals per (cell,
// velocity), the face records of the block (normal, S/V and upwind source per face), S/V
// times the normal of every in-block neighbour face, the cells' coefficient records; with
// `tc`, at least the tensor-core
// operand stage, which reuses it after the relaxation), then the chunk's velocities and
// weights, the in-block neighbour table and the tensor-core control words.
// `tc`: an FP32 gas sweep with Geom::tc set.
__host__ __device__ constexpr int sweep_nf_stride(int dim) { return dim < 3 ? 2 : 3; }
// rows of the diagonal area: one per cell; the FP64 gas sweep's moment basis takes up to 13
__host__ __device__ constexpr int sweep_diag_rows(int block, int planes, int dim, size_t real_size) {
    return planes == 4 && real_size == 8 && block < (dim < 3 ? 8 : 13) ? (dim < 3 ? 8 : 13) : block;
}
__host__ __device__ constexpr size_t sweep_face_bytes(int block, int dim, size_t real_size) {
    return (size_t)block * MAXF * 4 * real_size +
           ((size_t)block * MAXF * sweep_nf_stride(dim) * real_size + 31) / 32 * 32 + (size_t)block * cf::NC * real_size;
}

constexpr int NO_FACE = -2147483647 - 1;
__host__ __device__ constexpr size_t sweep_main_bytes(int block, int planes, int dim, size_t real_size, bool tc) {
    const size_t n = (size_t)(block * planes + sweep_diag_rows(block, planes, dim, real_size)) * SV * real_size +
                     sweep_face_bytes(block, dim, real_size);
    return tc && n < (size_t)tcm::STAGE_BYTES ? (size_t)tcm::STAGE_BYTES : n;
}

// One CTA = one relaxation block of consecutive cells x SV discrete velocities (N = 4 gas
// planes) or photon directions (N = 1); thread (tx, ty) = (velocity, row), and the
// block's cells are dealt to the SROWS rows round-robin.
//  0. the block's face records and in-block neighbour tables, staged in shared memory by
//     all threads at once;
//  1. residual and diagonal of every (cell, velocity) at f^k, independently: upwind
//     face values are the cell's own reconstruction on outflow faces and the
//     neighbour's (or the boundary state) on inflow faces;
//  2. forward and backward Gauss-Seidel inside the block with the first-order
//     operator, one thread per velocity (row 0);
//  3. f^{k+1/2} = f^k + delta, staged in shared memory;
//  4. velocity moments per (cell, chunk), eight lanes per cell.
// CL > 1: a cluster of CL CTAs takes the block.  Its cells are dealt to the rows of all of
// them; the residuals go to the first CTA's shared memory, which relaxes, and every CTA
// updates and sums its own cells.
template <typename Real, int N, int DIM, int ORDER, bool RESID = false, int ROWS = SROWS, int CL = 1>
__global__ void __launch_bounds__(SV * ROWS, sizeof(Real) == 4 ? (DIM < 3 ? 8 : 6) : 1) k_sweep(Geom<Real> g, Quad<Real> q, const Real *__restrict__ coef,
                                                      const Real *__restrict__ bcoef, const Real *__restrict__ f_in,
                                                      const Real *__restrict__ fface, Real *__restrict__ f_out,
                                                      Real *__restrict__ partial) {
    constexpr bool PHOTON = (N == 1);
    extern __shared__ unsigned char smem_raw[];
    Vec<Real, N> *R = reinterpret_cast<Vec<Real, N> *>(smem_raw);       // [block][SV]
    Real *Dg = reinterpret_cast<Real *>(R + g.block * SV);              // [block][SV] 1 / diagonal
    // [block][MAXF] face records: (n_x, n_y, S/V, source) in 1-D and 2-D, (S/V n, source) in 3-D
    Vec<Real, 4> *Fa = reinterpret_cast<Vec<Real, 4> *>(Dg + sweep_diag_rows(g.block, N, DIM, sizeof(Real)) * SV);
    constexpr int NFS = sweep_nf_stride(DIM);
    Real *Nf = reinterpret_cast<Real *>(Fa + g.block * MAXF);           // [block][MAXF][NFS] S/V n, in-block faces
    Real *sC = reinterpret_cast<Real *>(reinterpret_cast<unsigned char *>(Nf) +
                                        ((size_t)g.block * MAXF * NFS * sizeof(Real) + 31) / 32 * 32);   // [block][NC]
    // the tensor-core epilogue's basis covers the 1-D and 2-D moments
    constexpr bool tc = std::is_same<Real, float>::value && N == 4;
    static_assert(!tc || (DIM < 3 && !RESID), "FP32 gas without the tensor cores is k_sweep_gas32's");
    constexpr int NMPD = Lay<DIM>::NMP;
    Real *sxi = reinterpret_cast<Real *>(smem_raw + sweep_main_bytes(g.block, N, DIM, sizeof(Real), tc));   // [DIM+1][SV]
    signed char *Lg = reinterpret_cast<signed char *>(sxi + (DIM + 1) * SV);   // [block][MAXF] in-block neighbour or -1
    tcm::Ctl *ctl = reinterpret_cast<tcm::Ctl *>(Lg + ((g.block * MAXF + 15) & ~15));
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int rank = CL > 1 ? blockIdx.x % CL : 0, row0 = rank * ROWS + ty;
    const int c0 = blockIdx.x / CL * g.block;
    auto barrier = [] {
        if constexpr (CL > 1) cooperative_groups::this_cluster().sync();
        else __syncthreads();
    };
    // where the residuals and diagonals are relaxed
    Vec<Real, N> *Rr = R;
    Real *Dr = Dg;
    if constexpr (CL > 1 && !RESID) {
        Rr = cooperative_groups::this_cluster().map_shared_rank(R, 0);
        Dr = cooperative_groups::this_cluster().map_shared_rank(Dg, 0);
    }
    const int nb = min(g.block, g.n_cells - c0);
    const int chunk = blockIdx.y;
    const int v = chunk * SV + tx;
    const int stride = q.n_pad;
    // FP64: a warp of padding velocities alone leaves f as it is
    const bool idle = std::is_same<Real, double>::value && chunk * SV + (tx & 32) >= q.n;
    Real xi[DIM];
#pragma unroll
    for (int a = 0; a < DIM; ++a) xi[a] = q.x[a * stride + v];
    if (ty == 0) {
#pragma unroll
        for (int a = 0; a < DIM; ++a) sxi[a * SV + tx] = xi[a];
        sxi[DIM * SV + tx] = q.w[v];
    }
    if constexpr (tc) tcm::start(ctl, ty * SV + tx);   // the allocation completes during phase 1

    // ---- 0. face records: source = interior face id (order 2) or neighbour cell (order 1),
    // -1 - boundary face, NO_FACE past the cell's faces
    for (int t = ty * SV + tx; t < nb * MAXF; t += SV * ROWS) {
        const int l = t / MAXF, k = t - l * MAXF, i = c0 + l;
        Vec<Real, 4> fa;
        int lj = -1;
        if (k < g.info[i].x) {
            const Face<Real> F = load_face<Real, DIM>(g.fgeo, i, k);
            const int2 nb2 = g.fnb[i * MAXF + k];
            const int src = ORDER == 2 ? g.cface[i * MAXF + k] : nb2.x;
            if constexpr (DIM < 3) {
                fa.v[0] = F.n[0];
                fa.v[1] = DIM > 1 ? F.n[1] : Real(0);
                fa.v[2] = F.sv;
            } else {
                fa.v[0] = F.sv * F.n[0];
                fa.v[1] = F.sv * F.n[1];
                fa.v[2] = F.sv * F.n[2];
            }
            fa.v[3] = int_bits_as(src, Real(0));
            lj = nb2.y;
            if (lj >= 0) {
#pragma unroll
                for (int a = 0; a < NFS; ++a) Nf[t * NFS + a] = a < DIM ? F.sv * F.n[a] : Real(0);
            }
        } else {
            fa.v[0] = fa.v[1] = fa.v[2] = Real(0);
            fa.v[3] = int_bits_as(NO_FACE, Real(0));
        }
        Fa[t] = fa;
        Lg[t] = (signed char)lj;
    }
    // the block's coefficient records (gas planes; the photon plane reads two words per
    // cell): consecutive cells, one contiguous run
    if constexpr (!PHOTON)
        for (int t = ty * SV + tx; t < nb * (cf::NC / 4); t += SV * ROWS)
            reinterpret_cast<Vec<Real, 4> *>(sC)[t] = vload<Real, 4>(coef + (size_t)c0 * cf::NC + 4 * t);
    barrier();      // a cluster's CTAs have all started before one writes to another's shared memory

    // ---- 1. residuals and diagonals.  A cell's loads (its own value and the interior faces'
    // values: order 2 the face's upwind value, whichever side wrote it; order 1 the
    // neighbour's) are issued before its reference distribution, and for the single photon
    // plane, whose registers allow it, one cell ahead.
    auto issue = [&](int l, V<Real, N> &fi, V<Real, N> (&fk)[MAXF]) {
        fi = ldv<Real, N>(f_in, (size_t)(c0 + l) * stride + v);
#pragma unroll
        for (int k = 0; k < MAXF; ++k) {
            const int src = bits_as_int(Fa[l * MAXF + k].v[3]);
            if (src >= 0)
                fk[k] = ldv<Real, N>(ORDER == 2 ? fface : f_in, (size_t)src * stride + v);
            else
                fk[k] = vsplat<Real, N>(Real(0));
        }
    };
    constexpr bool AHEAD = PHOTON;
    V<Real, N> fi_next, fk_next[MAXF];
    if (AHEAD && row0 < nb) issue(row0, fi_next, fk_next);
    for (int l = row0; l < nb; l += CL * ROWS) {
        if (idle) {
            Rr[l * SV + tx] = Vec<Real, N>{};
            Dr[l * SV + tx] = Real(1);
            continue;
        }
        const Real *C = PHOTON ? coef + (size_t)(c0 + l) * cf::NC : sC + l * cf::NC;
        V<Real, N> fi, fk[MAXF];
        if constexpr (AHEAD) {
            fi = fi_next;
#pragma unroll
            for (int k = 0; k < MAXF; ++k) fk[k] = fk_next[k];
            if (l + CL * ROWS < nb) issue(l + CL * ROWS, fi_next, fk_next);
        } else {
            issue(l, fi, fk);
        }
        V<Real, N> r;
        const Vec<Real, 4> cc = vload<Real, 4>(C + cf::RATE);
        Real d;
        if constexpr (PHOTON) {
            const Real keff = vload<Real, 4>(C + cf::KEFF).v[0];
            r.x[0] = keff * (cc.v[3] - fi.x[0]);
            d = cc.v[1] + keff;
        } else {
            Real gp[4];
            reference<Real, DIM>(C, xi, gp);
            const Real rate = cc.v[0];
#pragma unroll
            for (int p = 0; p < 4; ++p) r.x[p] = (gp[p] - fi.x[p]) * rate;
            r.x[3] = fma(cc.v[2], fi.x[0], r.x[3]);
            d = cc.v[1] + rate;
        }
#pragma unroll
        for (int k = 0; k < MAXF; ++k) {
            const Vec<Real, 4> fa = Fa[l * MAXF + k];
            const int src = bits_as_int(fa.v[3]);
            if (src == NO_FACE) continue;
            // xn: xi . n (1-D, 2-D) or S/V xi . n (3-D); a: S/V xi . n
            Real xn = xi[0] * fa.v[0];
            if constexpr (DIM > 1) xn = fma(xi[1], fa.v[1], xn);
            if constexpr (DIM > 2) xn = fma(xi[2], fa.v[2], xn);
            if (is_zero(xn)) continue;
            const bool leaves = sizeof(Real) == 8 ? !is_neg(xn) : xn > Real(0);
            if (leaves) {
                if constexpr (DIM < 3) d = fma(fa.v[2], xn, d);
                else d += xn;
            }
            V<Real, N> fv;
            if (src >= 0 && (ORDER == 2 || !leaves)) {
                fv = fk[k];
            } else if (leaves) {
                fv = fi;
            } else if (g.bf_tab[-1 - src] >= 0) {
                // mirror plane: what enters at this velocity leaves at its mirror image
                const int t = g.bf_tab[-1 - src];
                const int vr = PHOTON ? g.refl_o[(size_t)t * stride + v] : g.refl_v[(size_t)t * stride + v];
                fv = ldv<Real, N>(f_in, (size_t)(c0 + l) * stride + vr);
            } else {
                const Real *B = bcoef + (size_t)(-1 - src) * bc::NB;
                if constexpr (PHOTON) {
                    fv.x[0] = B[bc::IIN];
                } else {
                    Real c2 = Real(0);
#pragma unroll
                    for (int a = 0; a < DIM; ++a) {
                        const Real c = xi[a] - B[bc::U + a];
                        c2 = fma(c, c, c2);
                    }
                    Real E;
                    if constexpr (sizeof(Real) == 8) E = B[bc::A] * fp64::exp_d(-B[bc::B] * c2);
                    else E = B[bc::A] * fexp(-B[bc::B] * c2);
                    fv.x[0] = E * B[bc::M0];
                    fv.x[1] = E * B[bc::MH];
                    fv.x[2] = E * B[bc::M1];
                    fv.x[3] = E * B[bc::M2];
                }
            }
            vfma(DIM < 3 ? -fa.v[2] * xn : -xn, fv, r);
        }
        Vec<Real, N> t;
#pragma unroll
        for (int p = 0; p < N; ++p) t.v[p] = r.x[p];
        Rr[l * SV + tx] = t;
        Dr[l * SV + tx] = rcp_r(d);          // the relaxation multiplies by 1/d
    }
    barrier();

    // ---- 2. Gauss-Seidel inside the block with the first-order operator; a = S/V xi_n from
    // the in-block face records of phase 0, used where a < 0 (in-block inflow):
    //   forward  delta*_l = (r_l - sum_{j<l} a delta*_j) / d_l
    //   backward delta_l  = delta*_l - (sum_{j>l} a delta_j) / d_l
    // (RESID: the residuals themselves are the result; phases 2 and 3 are skipped and
    // phase 4 takes their moments)
    if (ty == 0 && rank == 0 && !RESID && !idle) {
        for (int l = 0; l < nb; ++l) {
            Vec<Real, N> acc = R[l * SV + tx];
#pragma unroll
            for (int k = 0; k < MAXF; ++k) {
                const int lj = Lg[l * MAXF + k];
                if (lj < 0 || lj >= l) continue;
                Real a = Nf[(l * MAXF + k) * NFS] * xi[0];
                if constexpr (DIM > 1) a = fma(Nf[(l * MAXF + k) * NFS + 1], xi[1], a);
                if constexpr (DIM > 2) a = fma(Nf[(l * MAXF + k) * NFS + 2], xi[2], a);
                a = neg_part(a);        // outflow faces (a >= 0) add exactly nothing; no divergent branch
                const Vec<Real, N> dj = R[lj * SV + tx];
#pragma unroll
                for (int p = 0; p < N; ++p) acc.v[p] = fma(-a, dj.v[p], acc.v[p]);
            }
            const Real inv = Dg[l * SV + tx];
#pragma unroll
            for (int p = 0; p < N; ++p) acc.v[p] *= inv;
            R[l * SV + tx] = acc;
        }
        for (int l = nb - 1; l >= 0; --l) {
            Real corr[N];
#pragma unroll
            for (int p = 0; p < N; ++p) corr[p] = Real(0);
#pragma unroll
            for (int k = 0; k < MAXF; ++k) {
                const int lj = Lg[l * MAXF + k];
                if (lj <= l) continue;
                Real a = Nf[(l * MAXF + k) * NFS] * xi[0];
                if constexpr (DIM > 1) a = fma(Nf[(l * MAXF + k) * NFS + 1], xi[1], a);
                if constexpr (DIM > 2) a = fma(Nf[(l * MAXF + k) * NFS + 2], xi[2], a);
                a = neg_part(a);
                const Vec<Real, N> dj = R[lj * SV + tx];
#pragma unroll
                for (int p = 0; p < N; ++p) corr[p] = fma(a, dj.v[p], corr[p]);
            }
            Vec<Real, N> acc = R[l * SV + tx];
            const Real inv = Dg[l * SV + tx];
#pragma unroll
            for (int p = 0; p < N; ++p) acc.v[p] = fma(-corr[p], inv, acc.v[p]);
            R[l * SV + tx] = acc;
        }
    }
    barrier();

    // ---- 3. f^{k+1/2} = f^k + delta
    if constexpr (tc) {
        // Tensor-core moments: the tile's operand stage overlays R, the dead diagonal
        // and inflow areas and B; f^{k+1/2} waits in registers until every R read is done.
        unsigned char *stage = smem_raw;
        const int tile = c0 / MT * MT, lt0 = c0 - tile;
        constexpr int PER = MT / ROWS;
        Vec<float, 4> th[PER];
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int l = ty + j * ROWS;
            if (l < nb) {
                const size_t idx = (size_t)(c0 + l) * stride + v;
                const Vec<float, 4> fo = vload<float, 4>(reinterpret_cast<const float *>(f_in) + idx * 4);
                Vec<float, 4> t = *reinterpret_cast<const Vec<float, 4> *>(&R[l * SV + tx]);
#pragma unroll
                for (int p = 0; p < 4; ++p) t.v[p] += fo.v[p];
                if (g.pos_theta > 0.0f) {
#pragma unroll
                    for (int p = 0; p < 4; ++p) t.v[p] = fmaxf(t.v[p], g.pos_theta * fo.v[p]);
                }
                vstore<float, 4>(reinterpret_cast<float *>(f_out) + idx * 4, t);
                th[j] = t;
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int l = ty + j * ROWS;
            if (l < nb) tcm::put_a4(stage, lt0 + l, tx, th[j].v);
        }
        if (ty == 0) {
            const Vec<float, 4> u4 =
                vload<float, 4>(reinterpret_cast<const float *>(coef) + (size_t)tile * cf::NC + cf::U);
            float c[DIM];
#pragma unroll
            for (int a = 0; a < DIM; ++a) c[a] = (float)sxi[a * SV + tx] - u4.v[a];
            tcm::put_b<DIM>(stage, tx, c, (float)sxi[DIM * SV + tx]);
        }
        tcm::fence_smem_to_async();
        __syncthreads();
        // ---- 4. moments: one M = 128, N = 16, K = 64 contraction per CTA
        const int tid = ty * SV + tx;
        const uint32_t taddr = tcm::accumulator(ctl);
        float m[tcm::NBASIS];
        bool ok;
        if (tcm::contract(ctl, taddr, stage, tid, m, ok, g.tc_wait)) {
            const int l = (tid & 15) - lt0;
            if (l >= 0 && l < nb)
                tcm::store_row<DIM>(reinterpret_cast<float *>(partial) +
                                        ((size_t)(c0 + l) * gridDim.y + chunk) * NMPD,
                                    tid >> 5, m);
        }
        if (!ok && tid == 0) atomicOr(g.err, ERR_TIMEOUT_BIT);
        tcm::end(ctl, taddr, tid, ok, 0);
        return;
    }
    for (int l = row0; l < nb && !RESID; l += CL * ROWS) {
        const size_t idx = (size_t)(c0 + l) * stride + v;
        V<Real, N> fo = ldv<Real, N>(f_in, idx);
        Vec<Real, N> t = Rr[l * SV + tx];
#pragma unroll
        for (int p = 0; p < N; ++p) t.v[p] += fo.x[p];
        if (g.pos_theta > Real(0)) {   // the positivity bound of the implicit update
#pragma unroll
            for (int p = 0; p < N; ++p) t.v[p] = fmax(t.v[p], g.pos_theta * fo.x[p]);
        }
        R[l * SV + tx] = t;
        if constexpr (N == 1) {
            f_out[idx] = t.v[0];
        } else {
            vstore<Real, N>(f_out + idx * N, t);
        }
    }
    barrier();      // and the first CTA's residuals have been read

    // ---- 4. moments of the new distribution on CUDA cores, eight lanes per cell
    if constexpr (sizeof(Real) == 8 && !PHOTON) {
        // FP64: the basis w (1, c, cc, c|c|^2) of each velocity is formed once per moment tile
        // and chunk (over the dead diagonals), so that a value costs one instruction per
        // moment, and the eight lanes' sums are folded by halves (each lane keeps the half it
        // finishes), 21 additions instead of 51
        constexpr int NM = n_gas_moments<DIM>(), NB0 = 1 + DIM + DIM * (DIM + 1) / 2 + DIM;
        Real *bas = Dg;                                     // [NB0][SV]
        const int tid = ty * SV + tx, sub = tid & 7;
        for (int t0 = c0 / MT * MT; t0 < c0 + nb; t0 += MT) {
            if (t0 > c0) __syncthreads();
            if (ty == 0) {
                const Vec<Real, 4> u4 = vload<Real, 4>(coef + (size_t)t0 * cf::NC + cf::U);
                Real c[DIM], c2 = Real(0), wc[DIM];
                const Real w = sxi[DIM * SV + tx];
#pragma unroll
                for (int a = 0; a < DIM; ++a) {
                    c[a] = xi[a] - u4.v[a];
                    c2 = fma(c[a], c[a], c2);
                    wc[a] = w * c[a];
                }
                int m = 0;
                bas[m++ * SV + tx] = w;
#pragma unroll
                for (int a = 0; a < DIM; ++a) bas[m++ * SV + tx] = wc[a];
#pragma unroll
                for (int a = 0; a < DIM; ++a)
#pragma unroll
                    for (int b = a; b < DIM; ++b) bas[m++ * SV + tx] = wc[a] * c[b];
#pragma unroll
                for (int a = 0; a < DIM; ++a) bas[m++ * SV + tx] = wc[a] * c2;
            }
            __syncthreads();
            const int l0 = max(t0 - c0, 0), l1 = min(t0 + MT - c0, nb);
            for (int l = l0 + tid / 8; l < l1; l += SV * ROWS / 8) {
                if (CL > 1 && l / ROWS % CL != rank) continue;
                Real acc[24];
#pragma unroll
                for (int m = 0; m < 24; ++m) acc[m] = Real(0);
                for (int vl = sub; vl < SV; vl += 8) {
                    const Vec<Real, N> fv = R[l * SV + vl];
                    Real ph[NB0];
#pragma unroll
                    for (int b = 0; b < NB0; ++b) ph[b] = bas[b * SV + vl];
#pragma unroll
                    for (int b = 0; b < NB0; ++b) acc[b] = fma(ph[b], fv.v[0], acc[b]);
                    int m = NB0;
#pragma unroll
                    for (int p = (DIM < 3 ? 1 : 2); p < 4; ++p)
#pragma unroll
                        for (int b = 0; b <= DIM; ++b, ++m) acc[m] = fma(ph[b], fv.v[p], acc[m]);
                }
                fold8(acc, sub);
                Real *P = partial + ((size_t)(c0 + l) * gridDim.y + chunk) * NMPD;
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const int m = fold8_index(sub, q);
                    if (m < NM) P[m] = acc[q];
                }
            }
        }
        return;
    }
    if constexpr (PHOTON) {
        constexpr int TPC = 8;
        const int tid = ty * SV + tx;
        const int sub = tid % TPC;
        const unsigned gmask = 0xFFu << ((tid & 31) & ~(TPC - 1));
        for (int l = tid / TPC; l < nb; l += SV * ROWS / TPC) {
            Real acc[1 + DIM];
#pragma unroll
            for (int m = 0; m <= DIM; ++m) acc[m] = Real(0);
            for (int ol = sub; ol < SV; ol += TPC) {
                const Real wI = sxi[DIM * SV + ol] * R[l * SV + ol].v[0];
                acc[0] += wI;
#pragma unroll
                for (int a = 0; a < DIM; ++a) acc[1 + a] += wI * sxi[a * SV + ol];
            }
#pragma unroll
            for (int m = 0; m <= DIM; ++m)
#pragma unroll
                for (int s = 1; s < TPC; s <<= 1) acc[m] += __shfl_xor_sync(gmask, acc[m], s);
            if (sub == 0) {
                Real *P = partial + ((size_t)(c0 + l) * gridDim.y + chunk) * NMO;
#pragma unroll
                for (int m = 0; m <= DIM; ++m) P[m] = acc[m];
            }
        }
    }
}

// ------------------------------------------------------------------ the FP32 gas sweep
__device__ __forceinline__ float2 dup2(float x) { return make_float2(x, x); }
__device__ __forceinline__ float ex2(float x) {       // 2^x, subnormal results included
    float y;
    asm("ex2.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// 1 / x, one Newton step beyond rcp_normal
__device__ __forceinline__ float rcp_refined(float x) {
    const float y = rcp_normal(x);
    return fmaf(y, fmaf(-x, y, 1.0f), y);
}

// Shared memory of a k_sweep_gas32 CTA.
template <int DIM>
struct S32 {
    static constexpr int NK = (6 + 3 * DIM + 3) / 4;      // float4 of a Maxwellian: S B A A2 | K1 K2, then Q R1 R2 per axis
    static constexpr int CF = 2 + 3 * NK;                 // float4 of a cell's coefficients: u, Maxwellians, rates
    static constexpr int XS = DIM + 1;
    __host__ __device__ static constexpr size_t bytes(int block) {
        return (size_t)block * SV * 16                    // R: residuals, increments, f
               + (size_t)block * MAXF * 16                // face records
               + (size_t)block * MAXF * 16                // in-block neighbours
               + (size_t)block * CF * 16                  // coefficients
               + (size_t)block * SV * 4                   // 1 / diagonal
               + (size_t)XS * SV * 4                      // velocities and weights
               + ((size_t)block * 4 + 15) / 16 * 16;      // in-block neighbour counts
    }
};

// The reference distribution of the four planes at a pair of velocities (reference() above,
// with the second bracket as the first plus q.c).  A coefficient read from shared memory
// costs a register write per lane: it is read once for the pair, its products are scalar
// instructions, and what follows is packed.
template <int DIM>
__device__ __forceinline__ void reference32(const float4 *__restrict__ C, const float2 (&xi)[DIM], float2 (&gp)[4]) {
    constexpr int MH = 3 - DIM;
    const float4 u4 = C[0];
    const float uu[3] = {u4.x, u4.y, u4.z};
    float2 c[DIM], c2;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        c[a] = make_float2(xi[a].x - uu[a], xi[a].y - uu[a]);
        c2 = a == 0 ? __fmul2_rn(c[0], c[0]) : __ffma2_rn(c[a], c[a], c2);
    }
    auto mul = [](float s, float2 x) { return make_float2(s * x.x, s * x.y); };
    auto fma_ = [](float s, float2 x, float2 y) { return make_float2(fmaf(s, x.x, y.x), fmaf(s, x.y, y.y)); };
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float w[4 * S32<DIM>::NK];
#pragma unroll
        for (int t = 0; t < S32<DIM>::NK; ++t) {
            const float4 x = C[1 + k * S32<DIM>::NK + t];
            w[4 * t] = x.x;
            w[4 * t + 1] = x.y;
            w[4 * t + 2] = x.z;
            w[4 * t + 3] = x.w;
        }
        const float2 e = make_float2(ex2(w[0] * c2.x), ex2(w[0] * c2.y));
        float2 qc = mul(w[6], c[0]), r1 = mul(w[7], c[0]), r2 = mul(w[8], c[0]);
#pragma unroll
        for (int a = 1; a < DIM; ++a) {
            qc = fma_(w[6 + 3 * a], c[a], qc);
            r1 = fma_(w[7 + 3 * a], c[a], r1);
            r2 = fma_(w[8 + 3 * a], c[a], r2);
        }
        const float2 tb = make_float2(fmaf(w[1], c2.x, 0.5f * MH - 2.5f), fmaf(w[1], c2.y, 0.5f * MH - 2.5f));
        const float2 p0 = __ffma2_rn(qc, tb, dup2(1.0f)), E = mul(w[2], e);
        const float2 t1 = fma_(w[4], p0, r1), t2 = fma_(w[5], p0, r2);
        if (k == 0) {
            gp[0] = __fmul2_rn(E, p0);
            gp[1] = MH > 0 ? __fmul2_rn(mul(w[3], e), __fadd2_rn(p0, qc)) : dup2(0.0f);
            gp[2] = __fmul2_rn(E, t1);
            gp[3] = __fmul2_rn(E, t2);
        } else {
            gp[0] = __ffma2_rn(E, p0, gp[0]);
            if constexpr (MH > 0) gp[1] = __ffma2_rn(mul(w[3], e), __fadd2_rn(p0, qc), gp[1]);
            gp[2] = __ffma2_rn(E, t1, gp[2]);
            gp[3] = __ffma2_rn(E, t2, gp[3]);
        }
    }
}

// k_sweep for the four FP32 gas planes with CUDA-core moments: the same phases, a warp taking a
// cell's 64 velocities in pairs per lane, so that what is read for the cell is read once for
// both, without branches on the direction of a velocity.  FM: the most faces of a cell.
// It waits more than it works (43 % of the issue slots, L1 60 %, 3.3 TB/s): the relaxation,
// a serial chain over the block's cells in one warp, takes a quarter of the time (two warps of
// one velocity per lane, or reading ahead of it, took longer: more instructions).  Six CTAs of
// 80 registers per SM where no cell has more faces than a triangle, else five of 96 (at six,
// spills: 396 us; at four 358).  About 300 instructions per velocity, 497 before: 20 000
// triangles x 784 velocities at order 2 354 -> 292 us, 40 000 x 2 304 1.91 -> 1.56 ms, 10 185
// tetrahedra x 4 096 946 -> 814 us.
// ROWS: its warps; one where a block has no more than two cells, which leave the others without
// work and the SM without warps (10 000 tetrahedra x 1 728, blocks of one cell, order 1: 690 us
// with four, 241 with one; of two cells 403 and 172).
template <int DIM, int ORDER, bool RESID, int FM, int ROWS>
__global__ void __launch_bounds__(32 * ROWS, (FM < MAXF ? 24 : 20) / ROWS)
    k_sweep_gas32(Geom<float> g, Quad<float> q, const float *__restrict__ coef, const float *__restrict__ bcoef,
                  const float *__restrict__ f_in, const float *__restrict__ fface, float *__restrict__ f_out,
                  float *__restrict__ partial) {
    using S = S32<DIM>;
    constexpr int NT = 32 * ROWS;
    extern __shared__ float4 smem32[];
    float4 *R = smem32;                                   // [block][SV]
    float4 *Fa = R + g.block * SV;                        // [block][MAXF]: n, S/V (3-D: S/V n), source
    float4 *Gr = Fa + g.block * MAXF;                     // [block][MAXF]: S/V n, index; lower in-block neighbours from
                                                          // the front, upper ones from the back
    float4 *Cs = Gr + g.block * MAXF;                     // [block][CF]
    float *Dg = reinterpret_cast<float *>(Cs + g.block * S::CF);   // [block][SV]
    float *sxi = Dg + g.block * SV;                       // [DIM + 1][SV]
    int *Ln = reinterpret_cast<int *>(sxi + S::XS * SV);  // [block] lower + 8 upper in-block neighbours
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int c0 = blockIdx.x * g.block;
    const int nb = min(g.block, g.n_cells - c0);
    const int chunk = blockIdx.y;
    const int v = chunk * SV + tx;
    const int stride = q.n_pad;
    const unsigned row = (unsigned)stride * 16;
    const float *f_v = f_in + (size_t)v * 4;
    float2 xi[DIM];
#pragma unroll
    for (int a = 0; a < DIM; ++a) xi[a] = make_float2(q.x[a * stride + v], q.x[a * stride + v + 32]);

    // ---- 0. face records, in-block neighbours, coefficients
    for (int t = threadIdx.x; t < nb * MAXF; t += NT) {
        const int l = t / MAXF, k = t - l * MAXF, i = c0 + l, nf = g.info[i].x;
        float4 fa = make_float4(0.0f, 0.0f, 0.0f, __int_as_float(NO_FACE));
        int lj = -1, lower = 0, upper = 0, before = 0;
        float sn[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int m = 0; m < MAXF; ++m) {
            int o = m < nf ? g.fnb[i * MAXF + m].y : -1;
            if (o == l) o = -1;                           // a cell that is its own periodic neighbour
            lower += o >= 0 && o < l;
            upper += o > l;
            if (m == k) lj = o;
        }
#pragma unroll
        for (int m = 0; m < MAXF; ++m) {
            const int o = m < nf ? g.fnb[i * MAXF + m].y : -1;
            before += m < k && o >= 0 && o != l && (o < l) == (lj < l);
        }
        if (k < nf) {
            const Face<float> F = load_face<float, DIM>(g.fgeo, i, k);
            const int src = ORDER == 2 ? g.cface[i * MAXF + k] : g.fnb[i * MAXF + k].x;
#pragma unroll
            for (int a = 0; a < DIM; ++a) sn[a] = F.sv * F.n[a];
            if constexpr (DIM < 3) fa = make_float4(F.n[0], DIM > 1 ? F.n[1] : 0.0f, F.sv, __int_as_float(src));
            else fa = make_float4(sn[0], sn[1], sn[2], __int_as_float(src));
        }
        Fa[t] = fa;
        if (lj >= 0)
            Gr[l * MAXF + (lj < l ? before : MAXF - 1 - before)] = make_float4(sn[0], sn[1], sn[2], __int_as_float(lj));
        if (k == 0) Ln[l] = lower + 8 * upper;
    }
    for (int t = threadIdx.x; t < nb * 4; t += NT) {
        const int l = t >> 2, k = t & 3;
        const float *C = coef + (size_t)(c0 + l) * cf::NC;
        float4 *o = Cs + l * S::CF;
        if (k == 3) {
            o[0] = *reinterpret_cast<const float4 *>(C + cf::U);
            o[S::CF - 1] = *reinterpret_cast<const float4 *>(C + cf::RATE);
        } else {
            const float4 *P = reinterpret_cast<const float4 *>(C + cf::COMP + k * cf::CSZ);
            const float4 x0 = P[0], x1 = P[1], x2 = P[2], x3 = P[3];   // A B T K1 | Q K2 | R1 S | R2 A2
            const float Q[3] = {x1.x, x1.y, x1.z}, R1[3] = {x2.x, x2.y, x2.z}, R2[3] = {x3.x, x3.y, x3.z};
            float w[4 * S::NK];
            w[0] = x2.w;
            w[1] = x0.y;
            w[2] = x0.x;
            w[3] = x3.w;
            w[4] = x0.w;
            w[5] = x1.w;
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                w[6 + 3 * a] = Q[a];
                w[7 + 3 * a] = R1[a];
                w[8 + 3 * a] = R2[a];
            }
#pragma unroll
            for (int a = 6 + 3 * DIM; a < 4 * S::NK; ++a) w[a] = 0.0f;
#pragma unroll
            for (int a = 0; a < S::NK; ++a)
                o[1 + k * S::NK + a] = make_float4(w[4 * a], w[4 * a + 1], w[4 * a + 2], w[4 * a + 3]);
        }
    }
    for (int t = threadIdx.x; t < SV; t += NT) {
#pragma unroll
        for (int a = 0; a < DIM; ++a) sxi[a * SV + t] = q.x[a * stride + chunk * SV + t];
        sxi[DIM * SV + t] = q.w[chunk * SV + t];
    }
    __syncthreads();

    // ---- 1. residuals and diagonals; a cell's loads are issued before its reference
    for (int l = ty; l < nb; l += ROWS) {
        const float *nbr = (ORDER == 2 ? fface : f_in) + (size_t)v * 4;
        V<float, 4> fi[2], fk[FM][2], r[2];
        const float *own = row_at(f_v, c0 + l, row);
#pragma unroll
        for (int u = 0; u < 2; ++u) fi[u] = ldv<float, 4>(own, 32 * u);
#pragma unroll
        for (int k = 0; k < FM; ++k) {
            const int src = __float_as_int(Fa[l * MAXF + k].w);
            if (src < 0) continue;
            const float *p = row_at(nbr, src, row);
#pragma unroll
            for (int u = 0; u < 2; ++u) fk[k][u] = ldv<float, 4>(p, 32 * u);
        }
        float2 gp[4];
        reference32<DIM>(Cs + l * S::CF, xi, gp);
        const float4 cc = Cs[l * S::CF + S::CF - 1];      // rate, 1 / dt, sink
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            r[0].x[p] = (gp[p].x - fi[0].x[p]) * cc.x;
            r[1].x[p] = (gp[p].y - fi[1].x[p]) * cc.x;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) r[u].x[3] = fmaf(cc.z, fi[u].x[0], r[u].x[3]);
        float d[2] = {cc.y + cc.x, cc.y + cc.x};
#pragma unroll
        for (int k = 0; k < FM; ++k) {
            const float4 fa = Fa[l * MAXF + k];
            const int src = __float_as_int(fa.w);
            if (src == NO_FACE) continue;
            float a[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                a[u] = (u ? xi[0].y : xi[0].x) * fa.x;
                if constexpr (DIM > 1) a[u] = fmaf(u ? xi[1].y : xi[1].x, fa.y, a[u]);
                if constexpr (DIM > 2) a[u] = fmaf(u ? xi[2].y : xi[2].x, fa.z, a[u]);
                if constexpr (DIM < 3) {
                    d[u] = fmaf(fa.z, fmaxf(a[u], 0.0f), d[u]);
                    a[u] *= fa.z;
                } else {
                    d[u] += fmaxf(a[u], 0.0f);
                }
            }
            if (src >= 0) {
                // order 2: the face's upwind value serves both directions (a = 0: zero, never
                // written); order 1: the neighbour's value where it enters, the cell's where it
                // leaves (chosen, not multiplied by zero: a value that is not finite moves with
                // the flow only)
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    V<float, 4> up = fk[k][u];
                    if (ORDER == 1) {
#pragma unroll
                        for (int p = 0; p < 4; ++p) up.x[p] = a[u] < 0.0f ? up.x[p] : fi[u].x[p];
                    }
                    vfma(-a[u], up, r[u]);
                }
                continue;
            }
            const int bf = -1 - src, tab = g.bf_tab[bf];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                V<float, 4> fv;
                if (tab >= 0) {
                    // mirror plane: what enters at this velocity leaves at its mirror image
                    fv = ldv<float, 4>(row_at(f_in, c0 + l, row), g.refl_v[(size_t)tab * stride + v + 32 * u]);
                } else {
                    const float *B = bcoef + (size_t)bf * bc::NB;
                    float c2 = 0.0f;
#pragma unroll
                    for (int m = 0; m < DIM; ++m) {
                        const float c = (u ? xi[m].y : xi[m].x) - B[bc::U + m];
                        c2 = fmaf(c, c, c2);
                    }
                    const float E = B[bc::A] * fexp(-B[bc::B] * c2);
                    fv.x[0] = E * B[bc::M0];
                    fv.x[1] = E * B[bc::MH];
                    fv.x[2] = E * B[bc::M1];
                    fv.x[3] = E * B[bc::M2];
                }
                vfma(-fminf(a[u], 0.0f), fv, r[u]);
                vfma(-fmaxf(a[u], 0.0f), fi[u], r[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            R[l * SV + tx + 32 * u] = make_float4(r[u].x[0], r[u].x[1], r[u].x[2], r[u].x[3]);
            Dg[l * SV + tx + 32 * u] = rcp_refined(d[u]);
        }
    }
    __syncthreads();

    // ---- 2. Gauss-Seidel inside the block, one warp; the neighbour just relaxed stays in
    // registers.  The other warps meanwhile load f for phase 3.
    const float *R1 = reinterpret_cast<const float *>(R);
    constexpr int PRE = 2;                                // cells of phase 3 loaded ahead
    V<float, 4> fo[PRE][2];
    auto load_f = [&](int l, V<float, 4> (&x)[2]) {
#pragma unroll
        for (int u = 0; u < 2; ++u) x[u] = ldv<float, 4>(row_at(f_v, c0 + l, row), 32 * u);
    };
    auto load_ahead = [&] {
#pragma unroll
        for (int j = 0; j < PRE; ++j)
            if (ty + j * ROWS < nb) load_f(ty + j * ROWS, fo[j]);
    };
    if (!RESID && ty != 0) load_ahead();
    if (!RESID && ty == 0) {
        auto entering = [&](const float4 &gr, float (&a)[2]) {        // min(S/V xi . n, 0)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                a[u] = (u ? xi[0].y : xi[0].x) * gr.x;
                if constexpr (DIM > 1) a[u] = fmaf(u ? xi[1].y : xi[1].x, gr.y, a[u]);
                if constexpr (DIM > 2) a[u] = fmaf(u ? xi[2].y : xi[2].x, gr.z, a[u]);
                a[u] = fminf(a[u], 0.0f);
            }
        };
        V<float, 4> prev[2];
        auto pass = [&](bool up) {
            const int step = up ? -1 : 1;
            int l = up ? nb - 1 : 0;
            for (int t = 0; t < nb; ++t, l += step) {
                const int n = up ? Ln[l] >> 3 : Ln[l] & 7;
                float inv[2];
                V<float, 4> own[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    inv[u] = Dg[l * SV + tx + 32 * u];
                    own[u] = ldv<float, 4>(R1, l * SV + tx + 32 * u);
                }
                if (n > 0) {
                    const float4 g0 = Gr[l * MAXF + (up ? MAXF - 1 : 0)];
                    const int lj = __float_as_int(g0.w);
                    if (lj != l - step) {
#pragma unroll
                        for (int u = 0; u < 2; ++u) prev[u] = ldv<float, 4>(R1, lj * SV + tx + 32 * u);
                    }
                    // up: the sum of a dq over the neighbours; else r minus it
                    V<float, 4> s[2] = {up ? vsplat<float, 4>(0.0f) : own[0], up ? vsplat<float, 4>(0.0f) : own[1]};
                    float a[2];
                    entering(g0, a);
#pragma unroll
                    for (int u = 0; u < 2; ++u) vfma(up ? a[u] : -a[u], prev[u], s[u]);
                    for (int e = 1; e < n; ++e) {
                        const float4 gr = Gr[l * MAXF + (up ? MAXF - 1 - e : e)];
                        entering(gr, a);
#pragma unroll
                        for (int u = 0; u < 2; ++u)
                            vfma(up ? a[u] : -a[u], ldv<float, 4>(R1, __float_as_int(gr.w) * SV + tx + 32 * u), s[u]);
                    }
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        if (up) {
                            prev[u] = own[u];
                            vfma(-inv[u], s[u], prev[u]);
                        } else {
                            prev[u] = vmul(s[u], vsplat<float, 4>(inv[u]));
                        }
                    }
                } else {
#pragma unroll
                    for (int u = 0; u < 2; ++u) prev[u] = up ? own[u] : vmul(own[u], vsplat<float, 4>(inv[u]));
                }
#pragma unroll
                for (int u = 0; u < 2; ++u)
                    R[l * SV + tx + 32 * u] = make_float4(prev[u].x[0], prev[u].x[1], prev[u].x[2], prev[u].x[3]);
            }
        };
        pass(false);
        pass(true);
        load_ahead();
    }
    __syncthreads();

    // ---- 3. f^{k+1/2} = f^k + delta
    if constexpr (!RESID) {
        auto update = [&](int l, const V<float, 4> (&x)[2]) {
            float *to = const_cast<float *>(row_at(f_out + (size_t)v * 4, c0 + l, row));
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                V<float, 4> t = vadd(ldv<float, 4>(R1, l * SV + tx + 32 * u), x[u]);
                if (g.pos_theta > 0.0f) {   // the positivity bound of the implicit update
#pragma unroll
                    for (int p = 0; p < 4; ++p) t.x[p] = fmaxf(t.x[p], g.pos_theta * x[u].x[p]);
                }
                const float4 o = make_float4(t.x[0], t.x[1], t.x[2], t.x[3]);
                R[l * SV + tx + 32 * u] = o;
                *reinterpret_cast<float4 *>(to + 128 * u) = o;
            }
        };
        V<float, 4> more[PRE][2];
        for (int l0 = ty; l0 < nb; l0 += PRE * ROWS) {
            const int l1 = l0 + PRE * ROWS;
#pragma unroll
            for (int j = 0; j < PRE; ++j)
                if (l1 + j * ROWS < nb) load_f(l1 + j * ROWS, more[j]);
#pragma unroll
            for (int j = 0; j < PRE; ++j)
                if (l0 + j * ROWS < nb) update(l0 + j * ROWS, fo[j]);
#pragma unroll
            for (int j = 0; j < PRE; ++j)
#pragma unroll
                for (int u = 0; u < 2; ++u) fo[j][u] = more[j][u];
        }
        __syncthreads();
    }

    // ---- 4. velocity moments per (cell, chunk), eight lanes per cell
    constexpr int NM = n_gas_moments<DIM>(), NB0 = 1 + DIM + DIM * (DIM + 1) / 2 + DIM, NMPD = Lay<DIM>::NMP;
    const int sub = threadIdx.x & 7;
    for (int l = threadIdx.x >> 3; l < nb; l += NT / 8) {
        const float4 u4 = *reinterpret_cast<const float4 *>(coef + (size_t)((c0 + l) / MT * MT) * cf::NC + cf::U);
        const float uu[3] = {u4.x, u4.y, u4.z};
        // lin: planes (F0, H0) and (f1, f2) times 1, c; hi: F0 times cc, c |c|^2
        float2 lin[DIM + 1][2];
        float hi[NB0 - 1 - DIM];
#pragma unroll
        for (int b = 0; b <= DIM; ++b) lin[b][0] = lin[b][1] = dup2(0.0f);
#pragma unroll
        for (int b = 0; b < NB0 - 1 - DIM; ++b) hi[b] = 0.0f;
#pragma unroll 2
        for (int vl = sub; vl < SV; vl += 8) {
            const float4 x = R[l * SV + vl];
            const float w = sxi[DIM * SV + vl];
            float c[DIM], c2 = 0.0f, wc[DIM];
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                c[a] = sxi[a * SV + vl] - uu[a];
                c2 = fmaf(c[a], c[a], c2);
            }
            const float2 p0 = __fmul2_rn(dup2(w), make_float2(x.x, x.y)), p1 = __fmul2_rn(dup2(w), make_float2(x.z, x.w));
            lin[0][0] = __fadd2_rn(lin[0][0], p0);
            lin[0][1] = __fadd2_rn(lin[0][1], p1);
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                lin[1 + a][0] = __ffma2_rn(dup2(c[a]), p0, lin[1 + a][0]);
                lin[1 + a][1] = __ffma2_rn(dup2(c[a]), p1, lin[1 + a][1]);
                wc[a] = p0.x * c[a];
            }
            int m = 0;
#pragma unroll
            for (int a = 0; a < DIM; ++a)
#pragma unroll
                for (int b = a; b < DIM; ++b, ++m) hi[m] = fmaf(wc[a], c[b], hi[m]);
#pragma unroll
            for (int a = 0; a < DIM; ++a, ++m) hi[m] = fmaf(wc[a], c2, hi[m]);
        }
        float acc[24];
        int m = 0;
#pragma unroll
        for (int b = 0; b <= DIM; ++b) acc[m++] = lin[b][0].x;
#pragma unroll
        for (int b = 0; b < NB0 - 1 - DIM; ++b) acc[m++] = hi[b];
#pragma unroll
        for (int p = (DIM < 3 ? 1 : 2); p < 4; ++p)
#pragma unroll
            for (int b = 0; b <= DIM; ++b) acc[m++] = p & 1 ? lin[b][p >> 1].y : lin[b][p >> 1].x;
#pragma unroll
        for (int b = NM; b < 24; ++b) acc[b] = 0.0f;
        fold8(acc, sub);
        float *P = partial + ((size_t)(c0 + l) * gridDim.y + chunk) * NMPD;
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            const int b = fold8_index(sub, t);
            if (b < NM) P[b] = acc[t];
        }
    }
}

// ------------------------------------------------------------------ moments only
template <typename Real, int DIM>
__global__ void __launch_bounds__(VCH) k_moments_gas(int n_cells, Quad<Real> vq, const Real *__restrict__ coef,
                                                      const Real *__restrict__ f, Real *__restrict__ partial) {
    // one warp per (cell, chunk); lanes stride the chunk's velocities
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * (VCH / 32) + warp;
    const int chunk = blockIdx.y;
    if (i >= n_cells) return;
    constexpr int NM = n_gas_moments<DIM>();
    const Real *C = coef + (size_t)(i / MT * MT) * cf::NC;   // the tile's shift velocity
    constexpr int NMPD = Lay<DIM>::NMP;
    Real acc[NMPD];
#pragma unroll
    for (int m = 0; m < NMPD; ++m) acc[m] = Real(0);
    for (int vl = lane; vl < VCH; vl += 32) {
        const int v = chunk * VCH + vl;
        const Vec<Real, 4> fv4 = vload<Real, 4>(f + ((size_t)i * vq.n_pad + v) * 4);
        Real fv[4] = {fv4.v[0], fv4.v[1], fv4.v[2], fv4.v[3]};
        Real c[DIM];
#pragma unroll
        for (int a = 0; a < DIM; ++a) c[a] = vq.x[a * vq.n_pad + v] - C[cf::U + a];
        add_moments<Real, DIM>(acc, c, vq.w[v], fv);
    }
#pragma unroll
    for (int m = 0; m < NM; ++m)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[m] += __shfl_xor_sync(0xffffffffu, acc[m], o);
    if (lane == 0) {
        Real *P = partial + ((size_t)i * gridDim.y + chunk) * NMPD;
#pragma unroll
        for (int m = 0; m < NM; ++m) P[m] = acc[m];
    }
}

// FP64 moments: one warp per (MG cells of one moment tile, chunk of 64 velocities).  A lane's
// two velocities' basis w (1, c, cc, c|c|^2) is formed once for the MG cells, so that a value
// costs one FP64 instruction per moment, and the lanes' sums are folded by halves: 67 FP64
// instructions per (cell, chunk) in 2-D instead of 150 (2 048 cells x 784 velocities: 230 ->
// 109 us).
constexpr int MG = 4;
static_assert(MT % MG == 0, "a group lies in one moment tile");
template <int DIM>
struct MomentBasis {
    static constexpr int NM = n_gas_moments<DIM>(), NB0 = 1 + DIM + DIM * (DIM + 1) / 2 + DIM;
    double b[2][NB0];
    __device__ __forceinline__ MomentBasis(const Quad<double> &vq, int v0, int lane, const double *u) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int v = v0 + lane + 32 * h;
            const double w = vq.w[v];
            double c[DIM], wc[DIM], c2 = 0.0;
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                c[a] = vq.x[a * vq.n_pad + v] - u[a];
                c2 = fma(c[a], c[a], c2);
                wc[a] = w * c[a];
            }
            int m = 0;
            b[h][m++] = w;
#pragma unroll
            for (int a = 0; a < DIM; ++a) b[h][m++] = wc[a];
#pragma unroll
            for (int a = 0; a < DIM; ++a)
#pragma unroll
                for (int e = a; e < DIM; ++e) b[h][m++] = wc[a] * c[e];
#pragma unroll
            for (int a = 0; a < DIM; ++a) b[h][m++] = wc[a] * c2;
        }
    }
    // the moments of one cell's values at the lane's two velocities, summed over the warp
    __device__ __forceinline__ void store(const Vec<double, 4> (&f)[2], int lane, double *P) const {
        double acc[24];
#pragma unroll
        for (int m = 0; m < 24; ++m) acc[m] = 0.0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
            for (int k = 0; k < NB0; ++k) acc[k] = h ? fma(b[h][k], f[h].v[0], acc[k]) : b[h][k] * f[h].v[0];
            int m = NB0;
#pragma unroll
            for (int p = (DIM < 3 ? 1 : 2); p < 4; ++p)
#pragma unroll
                for (int k = 0; k <= DIM; ++k, ++m) acc[m] = h ? fma(b[h][k], f[h].v[p], acc[m]) : b[h][k] * f[h].v[p];
        }
        fold8(acc, lane & 7);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], 8);
            acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], 16);
            const int m = fold8_index(lane & 7, q);
            if (lane < 8 && m < NM) P[m] = acc[q];
        }
    }
};
template <int DIM>
__global__ void __launch_bounds__(VCH) k_moments_gas64(int n_cells, Quad<double> vq, const double *__restrict__ coef,
                                                        const double *__restrict__ f, double *__restrict__ partial) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i0 = (blockIdx.x * (VCH / 32) + warp) * MG, chunk = blockIdx.y;
    if (i0 >= n_cells) return;
    const MomentBasis<DIM> basis(vq, chunk * VCH, lane, coef + (size_t)(i0 / MT * MT) * cf::NC + cf::U);
    for (int i = i0; i < min(i0 + MG, n_cells); ++i) {
        const double *fp = f + ((size_t)i * vq.n_pad + chunk * VCH + lane) * 4;
        const Vec<double, 4> x[2] = {vload<double, 4>(fp), vload<double, 4>(fp + 128)};
        basis.store(x, lane, partial + ((size_t)i * gridDim.y + chunk) * Lay<DIM>::NMP);
    }
}

template <typename Real, int DIM>
__global__ void k_moments_photon(int n_cells, Quad<Real> oq, const Real *__restrict__ I, Real *__restrict__ partial) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * (blockDim.x / 32) + warp;
    const int chunk = blockIdx.y;
    if (i >= n_cells) return;
    Real acc[1 + DIM];
#pragma unroll
    for (int m = 0; m <= DIM; ++m) acc[m] = Real(0);
    for (int ol = lane; ol < OCH; ol += 32) {
        const int o = chunk * OCH + ol;
        const Real wI = oq.w[o] * I[(size_t)i * oq.n_pad + o];
        acc[0] += wI;
#pragma unroll
        for (int a = 0; a < DIM; ++a) acc[1 + a] += wI * oq.x[a * oq.n_pad + o];
    }
#pragma unroll
    for (int m = 0; m <= DIM; ++m)
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) acc[m] += __shfl_xor_sync(0xffffffffu, acc[m], s);
    if (lane == 0) {
        Real *P = partial + ((size_t)i * gridDim.y + chunk) * NMO;
#pragma unroll
        for (int m = 0; m <= DIM; ++m) P[m] = acc[m];
    }
}

// ------------------------------------------------------------------ GSIS synchronisation
// f <- f + w [f_eq(M_new) - f_eq(M_half)] with multi-temperature equilibria (planes
// F0, m T_t F0, d_r/2 T_r F0, d_v/2 T_v F0), fused with the moments of the result about
// the coefficient velocity; one warp per (cell, chunk).  Padding velocities are left alone.
template <typename Real, int DIM>
__global__ void __launch_bounds__(VCH) k_sync_gas(int n_cells, Quad<Real> vq, ModelDev m, double om,
                                                   const double *__restrict__ Fn, const double *__restrict__ Fh,
                                                   const Real *__restrict__ coef, Real *__restrict__ f,
                                                   Real *__restrict__ partial) {
    constexpr int MH = 3 - DIM;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * (VCH / 32) + warp;
    const int chunk = blockIdx.y;
    if (i >= n_cells) return;
    // The correction is the difference of two nearly equal Maxwellians near convergence.
    // It is evaluated as E_h [A_n expm1(-delta) + (A_n - A_h)] with
    // delta = B_n c_n^2 - B_h c_h^2 formed from per-cell differences taken in FP64, so that
    // its relative accuracy does not degrade as M^{k+1} -> M^{k+1/2}.  Where |delta| >= 1/2
    // the two Maxwellians differ by a large factor and are subtracted directly,
    // A_n exp(-B_h c_h^2 - delta) - A_h E_h: far out in velocity E_h underflows while
    // expm1(-delta) overflows, and their product would be 0 x inf.
    const double *rn = Fn + (size_t)i * NF, *rh = Fh + (size_t)i * NF;
    const double An = rn[0] * pow_neg_half_dim<DIM>(2.0 * 3.14159265358979323846 * rn[4]);
    const double Ah = rh[0] * pow_neg_half_dim<DIM>(2.0 * 3.14159265358979323846 * rh[4]);
    const double Bn = 0.5 / rn[4], Bh = 0.5 / rh[4];
    const double mn[4] = {1.0, MH * rn[4], 0.5 * m.d_r * rn[5], vib_energy<double>(m, rn[6])};
    const double mh[4] = {1.0, MH * rh[4], 0.5 * m.d_r * rh[5], vib_energy<double>(m, rh[6])};
    const Real An_r = (Real)An, dA = (Real)(An - Ah), Ah_r = (Real)Ah, Bn_r = (Real)Bn, Bh_r = (Real)Bh,
               dB = (Real)(Bn - Bh);
    Real uh[DIM], du[DIM], su[DIM], mul_n[4], dmul[4];
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        uh[a] = (Real)rh[1 + a];
        du[a] = (Real)(rh[1 + a] - rn[1 + a]);
        su[a] = (Real)(rh[1 + a] + rn[1 + a]);
    }
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        mul_n[p] = (Real)mn[p];
        dmul[p] = (Real)(mn[p] - mh[p]);
    }
    const Real w = (Real)om;
    constexpr int NM = n_gas_moments<DIM>();
    const Real *C = coef + (size_t)(i / MT * MT) * cf::NC;   // the tile's shift velocity
    constexpr int NMPD = Lay<DIM>::NMP;
    Real acc[NMPD];
#pragma unroll
    for (int k = 0; k < NMPD; ++k) acc[k] = Real(0);
    for (int vl = lane; vl < VCH; vl += 32) {
        const int v = chunk * VCH + vl;
        Real *fp = f + ((size_t)i * vq.n_pad + v) * 4;
        Vec<Real, 4> fv4 = vload<Real, 4>(fp);
        Real xi[DIM];
#pragma unroll
        for (int a = 0; a < DIM; ++a) xi[a] = vq.x[a * vq.n_pad + v];
        if (v < vq.n) {
            Real c2h = Real(0), dc2 = Real(0);
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                const Real ch = xi[a] - uh[a];
                c2h += ch * ch;
                dc2 += du[a] * (Real(2) * xi[a] - su[a]);    // c_n^2 - c_h^2
            }
            const Real Eh = fexp(-Bh_r * c2h);
            const Real delta = Bn_r * dc2 + dB * c2h;
            const Real e0h = Ah_r * Eh;                           // F0_h
            const Real d0 = fabs(delta) < Real(0.5) ? Eh * (An_r * expm1_r(-delta) + dA)
                                                    : An_r * fexp(-(Bh_r * c2h + delta)) - e0h;   // F0_n - F0_h
#pragma unroll
            for (int p = 0; p < 4; ++p) fv4.v[p] += w * (mul_n[p] * d0 + dmul[p] * e0h);
            vstore<Real, 4>(fp, fv4);
        }
        Real fv[4] = {fv4.v[0], fv4.v[1], fv4.v[2], fv4.v[3]};
        Real c[DIM];
#pragma unroll
        for (int a = 0; a < DIM; ++a) c[a] = xi[a] - C[cf::U + a];
        add_moments<Real, DIM>(acc, c, vq.w[v], fv);
    }
#pragma unroll
    for (int k = 0; k < NM; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
    if (lane == 0) {
        Real *P = partial + ((size_t)i * gridDim.y + chunk) * NMPD;
#pragma unroll
        for (int k = 0; k < NM; ++k) P[k] = acc[k];
    }
}

// ------------------------------------------------------------------ FP32 moments on tensor cores
// Per-cell constants of the synchronisation (see k_sync_gas), formed once per cell in FP64
// and rounded once: [0] A_n, [1] A_n - A_h, [2] A_h, [3] B_n, [4] B_h, [5] B_n - B_h,
// [6..] u_h, [6 + DIM..] u_h - u_n, [6 + 2 DIM..] u_h + u_n, [6 + 3 DIM..] the plane
// multipliers of M_n, [10 + 3 DIM..] their change; SKC floats per cell.
constexpr int SKC = SYNC_KC;
static_assert(SKC % 4 == 0, "constants are staged as float4");

template <int DIM>
__global__ void k_sync_coef(int n_cells, ModelDev m, const double *__restrict__ Fn, const double *__restrict__ Fh,
                            float *__restrict__ kc) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_cells) return;
    constexpr int MH = 3 - DIM;
    const double *rn = Fn + (size_t)i * NF, *rh = Fh + (size_t)i * NF;
    const double two_pi = 2.0 * 3.14159265358979323846;
    const double An = rn[0] * pow_neg_half_dim<DIM>(two_pi * rn[4]);
    const double Ah = rh[0] * pow_neg_half_dim<DIM>(two_pi * rh[4]);
    const double Bn = 0.5 / rn[4], Bh = 0.5 / rh[4];
    const double mn[4] = {1.0, MH * rn[4], 0.5 * m.d_r * rn[5], vib_energy<double>(m, rn[6])};
    const double mh[4] = {1.0, MH * rh[4], 0.5 * m.d_r * rh[5], vib_energy<double>(m, rh[6])};
    float K[SKC];
    for (int q = 0; q < SKC; ++q) K[q] = 0.f;
    K[0] = (float)An;
    K[1] = (float)(An - Ah);
    K[2] = (float)Ah;
    K[3] = (float)Bn;
    K[4] = (float)Bh;
    K[5] = (float)(Bn - Bh);
    for (int a = 0; a < DIM; ++a) {
        K[6 + a] = (float)rh[1 + a];
        K[6 + DIM + a] = (float)(rh[1 + a] - rn[1 + a]);
        K[6 + 2 * DIM + a] = (float)(rh[1 + a] + rn[1 + a]);
    }
    for (int p = 0; p < 4; ++p) {
        K[6 + 3 * DIM + p] = (float)mn[p];
        K[10 + 3 * DIM + p] = (float)(mn[p] - mh[p]);
    }
    for (int q = 0; q < SKC; ++q) kc[(size_t)i * SKC + q] = K[q];
}

constexpr int TC_SMEM = tcm::STAGE_BYTES + (int)sizeof(tcm::Ctl);

// Persistent, pipelined pass over the work items (moment tile of MT cells, chunk of 64
// velocities), one CTA of 128 threads per SM slot: thread (v = tid % 64, half = tid / 64)
// holds cells 8 * half .. 8 * half + 7 of a tile at velocity v.  While the tensor cores
// contract item k, the f loads of item k + 1 are in flight; the accumulator columns are
// allocated once per CTA and the completion barrier alternates phases.  SYNC: the
// synchronisation of k_sync_gas is applied to f (and stored) before the moments.
template <int DIM, bool SYNC>
__global__ void __launch_bounds__(128, 5) k_tc_pass(int n_cells, int n_chunks, int n_items, Quad<float> vq, float om,
                                                 const float4 *__restrict__ kc_g, const float *__restrict__ coef,
                                                 float *__restrict__ f, float *__restrict__ partial, int wait_limit,
                                                 int *__restrict__ err) {
    extern __shared__ __align__(1024) unsigned char tc_smem[];
    unsigned char *stage = tc_smem;
    tcm::Ctl *ctl = reinterpret_cast<tcm::Ctl *>(tc_smem + tcm::STAGE_BYTES);
    float4 *kc = reinterpret_cast<float4 *>(tc_smem + TC_SMEM);   // [MT][SKC / 4] (SYNC)
    const int tid = threadIdx.x, v = tid & 63, half = tid >> 6;
    tcm::start(ctl, tid);
    __syncthreads();
    const uint32_t taddr = tcm::accumulator(ctl);

    auto fetch = [&](int item, Vec<float, 4>(&x)[MT / 2]) {
        const int tile = item / n_chunks * MT, vg = (item % n_chunks) * tcm::K + v;
#pragma unroll
        for (int j = 0; j < MT / 2; ++j) {
            const int i = tile + half * (MT / 2) + j;
            x[j] = i < n_cells ? vload<float, 4>(f + ((size_t)i * vq.n_pad + vg) * 4) : Vec<float, 4>{};
        }
    };
    int item = blockIdx.x, prev = -1;
    uint32_t parity = 0;
    bool ok = true;
    // After a completion wait runs out (in any warp: the CTA agrees by a barrier vote)
    // the CTA issues no further chain, so that the one outstanding phase is the one
    // tcm::end waits for before it frees the accumulator.
    auto drain = [&](int it) {
        float m[tcm::NBASIS];
        bool okk;
        if (tcm::collect(ctl, taddr, tid, parity, m, okk, wait_limit)) {
            const int i = it / n_chunks * MT + (tid & 15);
            if (i < n_cells)
                tcm::store_row<DIM>(partial + ((size_t)i * n_chunks + it % n_chunks) * NMP, tid >> 5, m);
        }
        ok = __syncthreads_and(okk) != 0;
        parity ^= 1u;
    };
    Vec<float, 4> fv[MT / 2];
    if (item < n_items) fetch(item, fv);
    while (item < n_items) {
        const int next = item + gridDim.x;
        Vec<float, 4> fn[MT / 2];
        if (next < n_items) fetch(next, fn);              // in flight during the rest of the item
        if (prev >= 0) {
            drain(prev);
            if (!ok) break;
        }
        tcm::fence_before_sync();
        __syncthreads();                                   // accumulator read, stage free
        const int tile = item / n_chunks * MT, vg = (item % n_chunks) * tcm::K + v;
        if constexpr (SYNC) {
            if (tid < MT * (SKC / 4)) {
                const int i = tile + tid / (SKC / 4);
                kc[tid] = i < n_cells ? kc_g[(size_t)tile * (SKC / 4) + tid] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            __syncthreads();
            float xi[DIM];
#pragma unroll
            for (int a = 0; a < DIM; ++a) xi[a] = vq.x[a * vq.n_pad + vg];
#pragma unroll
            for (int j = 0; j < MT / 2; ++j) {
                const int l = half * (MT / 2) + j, i = tile + l;
                if (i < n_cells && vg < vq.n) {
                    // E_h [A_n expm1(-delta) + (A_n - A_h)], delta = B_n c_n^2 - B_h c_h^2, or
                    // the direct difference where |delta| >= 1/2 (as in k_sync_gas)
                    const float *Kc = reinterpret_cast<const float *>(kc + l * (SKC / 4));
                    float c2h = 0.f, dc2 = 0.f;
#pragma unroll
                    for (int a = 0; a < DIM; ++a) {
                        const float ch = xi[a] - Kc[6 + a];
                        c2h += ch * ch;
                        dc2 += Kc[6 + DIM + a] * (2.f * xi[a] - Kc[6 + 2 * DIM + a]);
                    }
                    const float Eh = fexp(-Kc[4] * c2h);
                    const float delta = Kc[3] * dc2 + Kc[5] * c2h;
                    const float e0h = Kc[2] * Eh;
                    const float d0 = fabsf(delta) < 0.5f ? Eh * (Kc[0] * expm1_r(-delta) + Kc[1])
                                                         : Kc[0] * fexp(-(Kc[4] * c2h + delta)) - e0h;
#pragma unroll
                    for (int p = 0; p < 4; ++p)
                        fv[j].v[p] += om * (Kc[6 + 3 * DIM + p] * d0 + Kc[10 + 3 * DIM + p] * e0h);
                    vstore<float, 4>(f + ((size_t)i * vq.n_pad + vg) * 4, fv[j]);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < MT / 2; ++j) tcm::put_a4(stage, half * (MT / 2) + j, v, fv[j].v);
        if (half == 0) {
            const Vec<float, 4> u4 = vload<float, 4>(coef + (size_t)tile * cf::NC + cf::U);
            float c[DIM];
#pragma unroll
            for (int a = 0; a < DIM; ++a) c[a] = vq.x[a * vq.n_pad + vg] - u4.v[a];
            tcm::put_b<DIM>(stage, v, c, vq.w[vg]);
        }
        tcm::fence_smem_to_async();
        __syncthreads();
        if (tid == 0) {
            tcm::fence_after_sync();
            tcm::issue(taddr, tcm::smem_u32(stage), tcm::smem_u32(&ctl->mbar));
        }
        prev = item;
        item = next;
#pragma unroll
        for (int j = 0; j < MT / 2; ++j) fv[j] = fn[j];
    }
    if (prev >= 0 && ok) drain(prev);
    if (!ok && tid == 0) atomicOr(err, ERR_TIMEOUT_BIT);
    tcm::end(ctl, taddr, tid, ok, parity ^ 1u);
}

// Grid of a persistent pass: every resident CTA slot of the device, at most one per item.
// The slots per SM follow from the kernel's registers and shared memory (the occupancy
// query reports a single CTA for kernels that allocate tensor memory); they are computed
// once per (instantiation, device) and cached, so that a launch costs no host-side query.
template <int DIM, bool SYNC>
static int persistent_grid(int smem, int n_items) {
    constexpr int MAXDEV = 64;
    static int slots[MAXDEV] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAXDEV) return n_items;
    if (slots[dev] == 0) {
        int sms = 0, smem_sm = 0, regs_sm = 0;
        cudaFuncAttributes fa;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev) != cudaSuccess ||
            cudaFuncGetAttributes(&fa, k_tc_pass<DIM, SYNC>) != cudaSuccess)
            return n_items;
        const int regs_cta = (fa.numRegs * 32 + 255) / 256 * 256 * 4;   // 4 warps, 256-register granules
        const int reserved = 1024;                                       // per-CTA system shared memory
        const int per = std::max(1, std::min({regs_sm / std::max(regs_cta, 1),
                                              smem_sm / (smem + (int)fa.sharedSizeBytes + reserved), 16}));
        slots[dev] = sms * per;
    }
    return std::max(1, std::min(n_items, slots[dev]));
}

template <typename Real, int DIM>
__global__ void k_sync_photon(int n_cells, Quad<Real> oq, ModelDev m, double om, const double *__restrict__ Fn,
                              const double *__restrict__ Fh, Real *__restrict__ I, Real *__restrict__ partial) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * (blockDim.x / 32) + warp;
    const int chunk = blockIdx.y;
    if (i >= n_cells) return;
    const double Tn = Fn[(size_t)i * NF + 7], Th = Fh[(size_t)i * NF + 7];
    const Real dI = (Real)(om * (m.sigma_R * Tn * Tn * Tn * Tn / 3.14159265358979323846 -
                                 m.sigma_R * Th * Th * Th * Th / 3.14159265358979323846));
    Real acc[1 + DIM];
#pragma unroll
    for (int k = 0; k <= DIM; ++k) acc[k] = Real(0);
    for (int ol = lane; ol < OCH; ol += 32) {
        const int o = chunk * OCH + ol;
        Real *ip = I + (size_t)i * oq.n_pad + o;
        Real x = *ip;
        if (o < oq.n) {
            x += dI;
            *ip = x;
        }
        const Real wI = oq.w[o] * x;
        acc[0] += wI;
#pragma unroll
        for (int a = 0; a < DIM; ++a) acc[1 + a] += wI * oq.x[a * oq.n_pad + o];
    }
#pragma unroll
    for (int k = 0; k <= DIM; ++k)
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], s);
    if (lane == 0) {
        Real *P = partial + ((size_t)i * gridDim.y + chunk) * NMO;
#pragma unroll
        for (int k = 0; k <= DIM; ++k) P[k] = acc[k];
    }
}

// ------------------------------------------------------------------ kinetic boundary fluxes
// Moments of the kinetic flux through every boundary face (one CTA per face): outgoing
// molecules carry the cell's distribution, incoming ones the wall Maxwellian (density
// from zero net mass flux of the outgoing ones) or the far-field state; photons likewise.
// Rows as the synthetic equations: mass, momentum, total energy, e_r, e_v, e_R.
// Rows of one boundary face from the velocity sums r: the outgoing part r[0..NS), the
// incoming unit-density part r[NS..2NS) scaled by the wall density (zero net mass flux) or
// the far-field density, and the photon flux r[2NS] (also added to the energy row).
template <int DIM>
__device__ __forceinline__ void kbflux_combine(const double *r, int kind, double rho_far, double *o) {
    constexpr int E = 1 + DIM, NS = DIM + 4;
    // wall: the density with zero net mass flux; far field: its density; mirror plane: the
    // incoming part is already in r[0..NS) (reflected cell values)
    const double scale = kind == 0 ? -r[0] / r[NS] : (kind == 1 ? rho_far : 0.0);
    for (int k = 0; k < NS; ++k) o[k] = r[k] + scale * r[NS + k];
    o[E + 3] = r[2 * NS];
    o[E] += o[E + 3];
}

template <typename Real, int DIM>
__global__ void __launch_bounds__(128) k_kinetic_bflux(MacroGeom g, ModelDev m, Quad<Real> vq, Quad<Real> oq,
                                                       const Real *__restrict__ f, const Real *__restrict__ I,
                                                       double *__restrict__ out, double *__restrict__ raw) {
    constexpr int MH = 3 - DIM, E = 1 + DIM, NS = DIM + 4;
    const int b = blockIdx.x;
    const int c = g.bf_cell[b];
    const int pid = g.bf_patch[b];
    const bool wall = g.patch_kind[pid] == 0;
    const int tab = g.bf_tab[b];     // >= 0: a mirror plane, entering values are the cell's mirror images
    const double *P = g.patch_state + (size_t)pid * 8;
    const double *n = g.bf_n + (size_t)b * MGS;
    const double T = P[4], Tr = wall ? P[4] : P[5], Tv = wall ? P[4] : P[6], TR = wall ? P[4] : P[7];
    const double Aw = pow_neg_half_dim<DIM>(2.0 * 3.14159265358979323846 * T), Bw = 0.5 / T;
    double acc[2 * NS + 1];
    for (int k = 0; k < 2 * NS + 1; ++k) acc[k] = 0.0;
    for (int v = threadIdx.x; v < vq.n; v += blockDim.x) {
        double xi[DIM], xn = 0.0, x2 = 0.0;
        for (int a = 0; a < DIM; ++a) {
            xi[a] = (double)vq.x[a * vq.n_pad + v];
            xn += xi[a] * n[a];
            x2 += xi[a] * xi[a];
        }
        const double wf = (double)vq.w[v] * xn;
        double f0, fh, f1, f2, *s;
        if (xn > 0.0) {
            const Vec<Real, 4> fv = vload<Real, 4>(f + ((size_t)c * vq.n_pad + v) * 4);
            f0 = fv.v[0];
            fh = fv.v[1];
            f1 = fv.v[2];
            f2 = fv.v[3];
            s = acc;
        } else if (tab >= 0) {
            const Vec<Real, 4> fv =
                vload<Real, 4>(f + ((size_t)c * vq.n_pad + g.refl_v[(size_t)tab * vq.n_pad + v]) * 4);
            f0 = fv.v[0];
            fh = fv.v[1];
            f1 = fv.v[2];
            f2 = fv.v[3];
            s = acc;
        } else {
            double c2 = 0.0;
            for (int a = 0; a < DIM; ++a) c2 += (xi[a] - P[1 + a]) * (xi[a] - P[1 + a]);
            f0 = Aw * exp(-Bw * c2);
            fh = MH * T * f0;
            f1 = 0.5 * m.d_r * Tr * f0;
            f2 = vib_energy<double>(m, Tv) * f0;
            s = acc + NS;
        }
        s[0] += wf * f0;
        for (int a = 0; a < DIM; ++a) s[1 + a] += wf * f0 * xi[a];
        s[E] += wf * (0.5 * x2 * f0 + 0.5 * fh + f1 + f2);
        s[E + 1] += wf * f1;
        s[E + 2] += wf * f2;
    }
    const double Iin = m.sigma_R * TR * TR * TR * TR / 3.14159265358979323846;
    for (int o = threadIdx.x; o < oq.n; o += blockDim.x) {
        double on = 0.0;
        for (int a = 0; a < DIM; ++a) on += (double)oq.x[a * oq.n_pad + o] * n[a];
        const double Iw = tab >= 0 ? (double)I[(size_t)c * oq.n_pad + g.refl_o[(size_t)tab * oq.n_pad + o]] : Iin;
        acc[2 * NS] += (double)oq.w[o] * on * (on > 0.0 ? (double)I[(size_t)c * oq.n_pad + o] : Iw);
    }
    __shared__ double buf[4][2 * NS + 1];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int k = 0; k < 2 * NS + 1; ++k) {
        double x = acc[k];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) buf[w][k] = x;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double r[2 * NS + 1];
        for (int k = 0; k < 2 * NS + 1; ++k) r[k] = buf[0][k] + buf[1][k] + buf[2][k] + buf[3][k];
        if (raw) {
            // velocity-sharded context: the sums over this rank's velocities, combined after
            // the sums over all ranks (k_kbflux_combine)
            for (int k = 0; k < KBR; ++k) raw[(size_t)b * KBR + k] = k < 2 * NS + 1 ? r[k] : 0.0;
            return;
        }
        kbflux_combine<DIM>(r, g.patch_kind[pid], P[0], out + (size_t)b * NVM);
    }
}

template <int DIM>
__global__ void k_kbflux_combine(MacroGeom g, const double *__restrict__ raw, double *__restrict__ out) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= g.n_bf) return;
    const int pid = g.bf_patch[b];
    kbflux_combine<DIM>(raw + (size_t)b * KBR, g.patch_kind[pid], g.patch_state[(size_t)pid * 8],
                        out + (size_t)b * NVM);
}

// ------------------------------------------------------------------ finish (FP64)
// Shifted moments S about the moment tile's velocity u0 (the velocity field of the
// tile's first cell, the shift every gas moment pass uses):
// with delta = S_c / rho the flow velocity is u0 + delta and every central moment
// follows from the binomial shift by delta.
// Sums of a cell's gas moment partials over the chunks first, first + step, ...: in FP32 two
// words per sum (Knuth's two-sum, the rounding error of every addition carried in the second
// word, itself summed plainly), off the slow FP64 pipe.  The fields stay within 1e-5 of the
// FP64 oracle from 13 chunks (784 velocities) up to 216 (13 824 velocities of the 3-D capsule)
// in the parity tests.
template <typename Real, int NM>
struct MomentSum {
    double s[NM];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int k = 0; k < NM; ++k) s[k] = 0.0;
    }
    __device__ __forceinline__ void add(int k, double x) { s[k] += x; }
    __device__ __forceinline__ double word(int k) const { return s[k]; }
    __device__ __forceinline__ void add_word(int k, double x) { s[k] += x; }
    __device__ __forceinline__ double value(int k) const { return s[k]; }
};
template <int NM>
struct MomentSum<float, NM> {
    float hi[NM], lo[NM];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int k = 0; k < NM; ++k) hi[k] = lo[k] = 0.0f;
    }
    __device__ __forceinline__ void add(int k, float b) {
        const float a = hi[k], t = a + b, bv = t - a;
        lo[k] += (a - (t - bv)) + (b - bv);
        hi[k] = t;
    }
    __device__ __forceinline__ float2 word(int k) const { return make_float2(hi[k], lo[k]); }
    __device__ __forceinline__ void add_word(int k, float2 x) {
        add(k, x.x);
        lo[k] += x.y;
    }
    __device__ __forceinline__ double value(int k) const { return to_double(hi[k]) + to_double(lo[k]); }
};
template <typename Real, int DIM>
__device__ __forceinline__ void sum_chunks(int i, int first, int step, int n_chunks, const Real *__restrict__ partial,
                                           MomentSum<Real, n_gas_moments<DIM>()> &S) {
    constexpr int NM = n_gas_moments<DIM>(), NMPD = Lay<DIM>::NMP;   // partial stride
    static_assert(NMPD % 4 == 0 && NM <= NMPD && NMO == 4 && DIM + 1 <= NMO, "partial records are read as 4-vectors");
    S.zero();
#pragma unroll 2
    for (int c = first; c < n_chunks; c += step) {
        const Real *P = partial + ((size_t)i * n_chunks + c) * NMPD;
#pragma unroll
        for (int q = 0; q < NMPD / 4; ++q) {
            const Vec<Real, 4> p4 = vload<Real, 4>(P + 4 * q);
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (4 * q + e < NM) S.add(4 * q + e, p4.v[e]);
        }
    }
}

template <typename Real, int DIM>
__device__ __forceinline__ void finish_cell(int i, int o_chunks, const ModelDev &m, const Real *__restrict__ coef,
                                            const MomentSum<Real, n_gas_moments<DIM>()> &sums,
                                            const Real *__restrict__ opartial, const double *__restrict__ vol,
                                            const double *__restrict__ F_old, double *__restrict__ F_new,
                                            double *__restrict__ eps_terms, int *__restrict__ err, int have_old,
                                            const double *__restrict__ X, double (&E)[NEPS]) {
    constexpr int NM = n_gas_moments<DIM>();
    constexpr int MH = 3 - DIM;
    double S[NM];
    double Ph[1 + DIM];
    if (X) {
        // per-cell sums of a velocity-sharded context, already summed over the ranks
        // (velocity shards are built for 1-D and 2-D)
        if constexpr (DIM < 3) {
            static_assert(DIM >= 3 || NM <= NMP, "exchange record");
#pragma unroll
            for (int k = 0; k < NM; ++k) S[k] = X[(size_t)i * NXC + k];
#pragma unroll
            for (int k = 0; k <= DIM; ++k) Ph[k] = X[(size_t)i * NXC + NMP + k];
        }
    } else {
#pragma unroll
        for (int k = 0; k < NM; ++k) S[k] = sums.value(k);
    }
    if (!X) {
#pragma unroll
        for (int k = 0; k <= DIM; ++k) Ph[k] = 0.0;
        for (int c = 0; c < o_chunks; ++c) {
            const Vec<Real, 4> p4 = vload<Real, 4>(opartial + ((size_t)i * o_chunks + c) * NMO);
#pragma unroll
            for (int k = 0; k <= DIM; ++k) Ph[k] += to_double(p4.v[k]);
        }
    }
    // unpack
    int k = 0;
    const double rho = S[k++];
    double Sc[DIM], Scc[DIM][DIM], Sc3[DIM];
    for (int a = 0; a < DIM; ++a) Sc[a] = S[k++];
    for (int a = 0; a < DIM; ++a)
        for (int b = a; b < DIM; ++b) {
            Scc[a][b] = S[k];
            Scc[b][a] = S[k];
            ++k;
        }
    for (int a = 0; a < DIM; ++a) Sc3[a] = S[k++];
    double H0 = 0.0, Hc[DIM];
    for (int a = 0; a < DIM; ++a) Hc[a] = 0.0;
    if (MH > 0) {
        H0 = S[k++];
        for (int a = 0; a < DIM; ++a) Hc[a] = S[k++];
    }
    const double G1 = S[k++];
    double G1c[DIM];
    for (int a = 0; a < DIM; ++a) G1c[a] = S[k++];
    const double G2 = S[k++];
    double G2c[DIM];
    for (int a = 0; a < DIM; ++a) G2c[a] = S[k++];

    // one reciprocal of rho; constants of the model as reciprocals (an FP64 division is nine
    // FP64 instructions, 64 cycles each)
    const double ir = rcp_r(rho);
    double dl[DIM];
    for (int a = 0; a < DIM; ++a) dl[a] = Sc[a] * ir;
    // central second moments  P_ab = int (c-d)_a (c-d)_b F0 = Scc_ab - rho d_a d_b
    double P[DIM][DIM], trP = 0.0;
    for (int a = 0; a < DIM; ++a)
        for (int b = 0; b < DIM; ++b) P[a][b] = Scc[a][b] - rho * dl[a] * dl[b];
    for (int a = 0; a < DIM; ++a) trP += P[a][a];
    const double int_c2 = trP + H0;                       // int c^2 f0 over all velocity components
    double *Fn = F_new + (size_t)i * NF;
    for (int q = 0; q < NF; ++q) Fn[q] = 0.0;
    const Real *C = coef + (size_t)(i / MT * MT) * cf::NC;   // the tile's shift velocity
    Fn[0] = rho;
    for (int a = 0; a < DIM; ++a) Fn[1 + a] = to_double(C[cf::U + a]) + dl[a];
    const double Tt = int_c2 * ((1.0 / 3.0) * ir);
    // the record's temperatures are read back from registers below, not from memory
    const double Tr = G1 * (m.i_half_dr * ir);
    const double Tv = m.dv_T ? vib_temperature<double>(m, G2 * ir) : G2 * (m.i_half_dv * ir);   // int f2 = d_v(T_v) rho T_v / 2
    Fn[4] = Tt;
    Fn[5] = Tr;
    Fn[6] = Tv;
    const double eR = Ph[0];
    Fn[7] = m.sigma_R > 0.0 ? sqrt_r(sqrt_r((is_neg(eR) ? 0.0 : eR) * m.i_4sigma)) : 0.0;
    // heat fluxes: q_t,a = 1/2 int (c-d)_a ((c-d)^2 F0 + H0)
    //   int (c-d)_a |c-d|^2 F0 = Sc3_a - 2 sum_b d_b Scc_ab - d_a trScc + |d|^2 Sc_a
    //                            + 2 d_a (d . Sc) - rho d_a |d|^2  (Sc = rho d)
    double trS = 0.0, d2 = 0.0, dSc = 0.0;
    for (int a = 0; a < DIM; ++a) {
        trS += Scc[a][a];
        d2 += dl[a] * dl[a];
        dSc += dl[a] * Sc[a];
    }
    for (int a = 0; a < DIM; ++a) {
        double t = Sc3[a] - dl[a] * trS + d2 * Sc[a] + 2.0 * dl[a] * dSc - rho * dl[a] * d2;
        for (int b = 0; b < DIM; ++b) t -= 2.0 * dl[b] * Scc[a][b];
        const double hflux = Hc[a] - dl[a] * H0;
        Fn[8 + a] = 0.5 * (t + hflux);
        Fn[11 + a] = G1c[a] - dl[a] * G1;
        Fn[14 + a] = G2c[a] - dl[a] * G2;
        Fn[17 + a] = Ph[1 + a];
    }
    // stress (xx, yy, zz, xy, xz, yz)
    double sig[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    for (int a = 0; a < DIM; ++a)
        for (int b = 0; b < DIM; ++b) sig[a][b] = P[a][b];
    for (int a = DIM; a < 3; ++a) sig[a][a] = MH > 0 ? H0 * (MH == 2 ? 0.5 : 1.0) : 0.0;
    for (int a = 0; a < 3; ++a) sig[a][a] -= int_c2 * (1.0 / 3.0);
    Fn[20] = sig[0][0];
    Fn[21] = sig[1][1];
    Fn[22] = sig[2][2];
    Fn[23] = sig[0][1];
    Fn[24] = sig[0][2];
    Fn[25] = sig[1][2];

    // positive and finite, by the bit patterns
    auto good = [](double x) { return (unsigned long long)__double_as_longlong(x) - 1ull < 0x7fefffffffffffffull; };
    const bool bad = !good(rho) || !good(Tt) || !good(Tr) || !good(Tv) ||
                     (__double2hiint(eR) & 0x7ff00000) == 0x7ff00000;
    if (bad) atomicOr(err, 1);
    // convergence terms: (drho^2, rho^2, |du|^2, |u|^2, dT^2, T^2, T) * V
    const double V = vol[i];
    // total temperature of Section 2.1: (3 + d_r + d_v(T)) T = 3 T_t + d_r T_r + d_v(T_v) T_v
    if (have_old) {
        const double Ttot = m.dv_T ? equal_temperature<double>(m, 3.0 + m.d_r, 3.0 * Tt + m.d_r * Tr +
                                                                                   2.0 * vib_energy<double>(m, Tv))
                                   : (3.0 * Tt + m.d_r * Tr + m.d_v * Tv) * m.i_heat;
        const double *Fo = F_old + (size_t)i * NF;
        const double To = m.dv_T ? equal_temperature<double>(m, 3.0 + m.d_r, 3.0 * Fo[4] + m.d_r * Fo[5] +
                                                                                 2.0 * vib_energy<double>(m, Fo[6]))
                                 : (3.0 * Fo[4] + m.d_r * Fo[5] + m.d_v * Fo[6]) * m.i_heat;
        double du2 = 0.0, uo2 = 0.0;
        for (int a = 0; a < DIM; ++a) {
            du2 += (Fn[1 + a] - Fo[1 + a]) * (Fn[1 + a] - Fo[1 + a]);
            uo2 += Fo[1 + a] * Fo[1 + a];
        }
        E[0] = (rho - Fo[0]) * (rho - Fo[0]) * V;
        E[1] = Fo[0] * Fo[0] * V;
        E[2] = du2 * V;
        E[3] = uo2 * V;
        E[4] = (Ttot - To) * (Ttot - To) * V;
        E[5] = To * To * V;
        E[6] = To * V;
        E[7] = 0.0;
    } else {
        for (int q = 0; q < NEPS; ++q) E[q] = 0.0;
    }
    for (int q = 0; q < NEPS; ++q) eps_terms[(size_t)i * NEPS + q] = E[q];
}

// One cell per lane of the first warp; FW warps share the sums over the chunks (from four
// chunks on: 10 000 cells x 36 chunks 39 -> 30 us, 20 000 x 13 34 -> 33).  With `reduce`, the
// convergence terms are summed too: each CTA adds its 32 cells in a fixed shuffle order, and
// the last CTA to finish (counted with an atomic ticket after a fence, no waiting) adds the
// CTA partials in a fixed order, so the result does not depend on scheduling.
template <typename Real, int DIM, int FW>
__global__ void __launch_bounds__(32 * FW) k_finish(int n_cells, int n_chunks, int o_chunks, ModelDev m,
                                                    const Real *__restrict__ coef, const Real *__restrict__ partial,
                                                    const Real *__restrict__ opartial, const double *__restrict__ vol,
                                                    const double *__restrict__ F_old, double *__restrict__ F_new,
                                                    double *__restrict__ eps_terms, int *__restrict__ err, int have_old,
                                                    int reduce, double *__restrict__ eps_part,
                                                    unsigned int *__restrict__ ticket, double *__restrict__ eps_sums,
                                                    const double *__restrict__ X) {
    constexpr int NM = n_gas_moments<DIM>();
    using Sum = MomentSum<Real, NM>;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane;
    Sum S;
    if (i < n_cells && !X) sum_chunks<Real, DIM>(i, w, FW, n_chunks, partial, S);
    if constexpr (FW > 1) {
        __shared__ double words[FW - 1][NM][32];     // a double, or the two FP32 words of a sum
        using Word = decltype(S.word(0));
        if (w > 0) {
#pragma unroll
            for (int k = 0; k < NM; ++k) *reinterpret_cast<Word *>(&words[w - 1][k][lane]) = S.word(k);
        }
        __syncthreads();
        if (w > 0) return;
#pragma unroll
        for (int v = 0; v < FW - 1; ++v)
#pragma unroll
            for (int k = 0; k < NM; ++k) S.add_word(k, *reinterpret_cast<const Word *>(&words[v][k][lane]));
    }
    double E[NEPS];
    for (int q = 0; q < NEPS; ++q) E[q] = 0.0;
    if (i < n_cells)
        finish_cell<Real, DIM>(i, o_chunks, m, coef, S, opartial, vol, F_old, F_new, eps_terms, err, have_old, X, E);
    if (!reduce) return;
#pragma unroll
    for (int q = 0; q < NEPS; ++q)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) E[q] += __shfl_xor_sync(0xffffffffu, E[q], o);
    bool last = false;
    if (lane == 0) {
        for (int q = 0; q < NEPS; ++q) eps_part[(size_t)blockIdx.x * NEPS + q] = E[q];
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    __threadfence();
    double acc[NEPS];
    for (int q = 0; q < NEPS; ++q) acc[q] = 0.0;
#pragma unroll 4
    for (int b = lane; b < (int)gridDim.x; b += 32)
#pragma unroll
        for (int q = 0; q < NEPS; ++q) acc[q] += __ldcg(eps_part + (size_t)b * NEPS + q);   // L2: other CTAs' writes
#pragma unroll
    for (int q = 0; q < NEPS; ++q)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
    if (lane == 0) {
        for (int q = 0; q < NEPS; ++q) eps_sums[q] = acc[q];
        *ticket = 0u;
    }
}

// ------------------------------------------------------------------ equilibrium
template <typename Real, int DIM>
__global__ void k_equilibrium(int n_cells, Quad<Real> vq, Quad<Real> oq, ModelDev m, const double *__restrict__ F,
                              Real *__restrict__ f, Real *__restrict__ I) {
    // 17 FP64 instructions per velocity (50 with a division, exp and conversions by
    // instruction): 20 000 cells x 784 velocities, FP32 storage, 1.36 -> 0.75 ms
    const int i = blockIdx.x;
    const double *M = F + (size_t)i * NF;
    const double rho = M[0], Tt = M[4];
    const double norm = rho * pow_neg_half_dim<DIM>(6.283185307179586 * Tt), sc = -fp64::EXP_SCALE / (2.0 * Tt);
    const double mh = (3 - DIM) * Tt, m1 = 0.5 * m.d_r * M[5], m2 = vib_energy<double>(m, M[6]);
    for (int v = threadIdx.x; v < vq.n_pad; v += blockDim.x) {
        double c2 = 0.0;
        for (int a = 0; a < DIM; ++a) {
            const double c = to_double(vq.x[a * vq.n_pad + v]) - M[1 + a];
            c2 = fma(c, c, c2);
        }
        const double F0 = norm * fp64::exp2n(sc, c2);
        Vec<Real, 4> t;
        t.v[0] = to_real<Real>(F0);
        t.v[1] = to_real<Real>(mh * F0);
        t.v[2] = to_real<Real>(m1 * F0);
        t.v[3] = to_real<Real>(m2 * F0);
        vstore<Real, 4>(f + ((size_t)i * vq.n_pad + v) * 4, t);
    }
    const double B = m.sigma_R * M[7] * M[7] * M[7] * M[7] / 3.141592653589793;
    for (int o = threadIdx.x; o < oq.n_pad; o += blockDim.x) I[(size_t)i * oq.n_pad + o] = (Real)B;
}

// ---- two-word FP32: a value as x + y with |y| at most about a unit of x's last place.  FP32
// storage needs its equilibria to FP32 rounding, which exp in FP32 alone does not give (its
// argument reaches 100); an FP64 instruction takes the time of some 70 of these.
__device__ __forceinline__ float2 two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), t = __fadd_rn(s, -a);
    return make_float2(s, __fadd_rn(__fadd_rn(a, -__fadd_rn(s, -t)), __fadd_rn(b, -t)));
}
__device__ __forceinline__ float2 two_sum_ordered(float a, float b) {   // |a| >= |b|
    const float s = __fadd_rn(a, b);
    return make_float2(s, __fadd_rn(b, -__fadd_rn(s, -a)));
}
__device__ __forceinline__ float2 two_diff(float x, float uh, float ul) {   // x - (uh + ul)
    const float2 d = two_sum(x, -uh);
    return make_float2(d.x, __fadd_rn(d.y, -ul));
}
__device__ __forceinline__ float2 square2(float2 d) {
    const float p = __fmul_rn(d.x, d.x);
    return make_float2(p, fmaf(__fadd_rn(d.x, d.x), d.y, fmaf(d.x, d.x, -p)));
}
__device__ __forceinline__ float2 add2w(float2 a, float2 b) {
    const float2 s = two_sum(a.x, b.x);
    return make_float2(s.x, __fadd_rn(s.y, __fadd_rn(a.y, b.y)));
}
// 2^(j / EXP2_N) in two words, built by the compiler from the table of fp64.cuh
constexpr int EXP2_N = 64;
struct Exp2Table {
    float hi[EXP2_N], lo[EXP2_N];
};
constexpr Exp2Table make_exp2_table() {
    constexpr fp64::ExpTable E = fp64::make_exp_table();
    Exp2Table T{};
    for (int j = 0; j < EXP2_N; ++j) {
        const double x = E.t[j * (fp64::EXP_N / EXP2_N)];
        T.hi[j] = (float)x;
        T.lo[j] = (float)(x - (double)T.hi[j]);
    }
    return T;
}
__constant__ const Exp2Table g_exp2_table = make_exp2_table();
// 2^(s c2) = v 2^k: 2^(j/EXP2_N) from the table times e^r, |r| <= ln 2 / (2 EXP2_N), by its
// Taylor sum.  The rounding of the sum's r^2/2 term is what the result is off by beyond its own
// rounding: 4e-5 units in the last place (2e-3 with EXP2_N = 8).
struct Exp2 {
    float2 v;
    float scale;       // v carries the other half of the exponent, so that both are normal numbers
};
__device__ __forceinline__ Exp2 exp2_two(const float2 *__restrict__ table, float2 s, float2 c2) {
    float y = __fmul_rn(s.x, c2.x), yl = fmaf(s.y, c2.x, fmaf(s.x, c2.y, fmaf(s.x, c2.x, -y)));
    if (fabsf(y) > 250.0f) {         // 0 or infinite in FP32
        y = copysignf(250.0f, y);
        yl = 0.0f;
    }
    const float k = rintf((float)EXP2_N * y), f = fmaf(-1.0f / EXP2_N, k, y);
    const float2 g = two_sum_ordered(f, yl);
    const float L = 0.693147182f, Ll = -1.90465421e-9f;      // ln 2
    const float r = __fmul_rn(g.x, L), rl = fmaf(g.y, L, fmaf(g.x, Ll, fmaf(g.x, L, -r)));
    const float p = fmaf(r, fmaf(r, 1.0f / 24.0f, 1.0f / 6.0f), 0.5f);
    const float2 q = two_sum_ordered(r, fmaf(__fmul_rn(r, r), p, rl));      // e^r - 1
    const int ki = (int)k, n = ki >> 6, n1 = n >> 1;
    static_assert(EXP2_N == 64, "the integer part is a shift by 6");
    const float2 T = table[ki & (EXP2_N - 1)];
    const float t = __fmul_rn(T.x, q.x);
    const float2 e = two_sum_ordered(T.x, t);
    const float el = __fadd_rn(e.y, fmaf(T.x, q.y, fmaf(T.y, q.x, __fadd_rn(T.y, fmaf(T.x, q.x, -t)))));
    const float s1 = __int_as_float((n1 + 127) << 23);
    Exp2 o;
    o.v = make_float2(__fmul_rn(e.x, s1), __fmul_rn(el, s1));
    o.scale = __int_as_float((n - n1 + 127) << 23);
    return o;
}
__device__ __forceinline__ float scaled(float2 N, const Exp2 &e) {   // (N 2^..) to FP32
    const float r = __fmul_rn(N.x, e.v.x);
    return __fmul_rn(__fadd_rn(r, fmaf(N.x, e.v.y, fmaf(N.y, e.v.x, fmaf(N.x, e.v.x, -r)))), e.scale);
}

// The equilibrium in FP32 storage: the start of a run writes f once, and in FP64 arithmetic
// (the kernel above) its time is that of 17 FP64 instructions per velocity.  Here each cell's
// constants are formed in FP64 by one thread and kept as two FP32 words, and a velocity takes
// about 100 FP32 instructions; a value is within 0.5001 units in the last place (0.5000 in FP64
// arithmetic).
template <int DIM>
__global__ void __launch_bounds__(256) k_equilibrium32(int n_cells, int cells, Quad<float> vq, Quad<float> oq,
                                                       ModelDev m, const double *__restrict__ F,
                                                       float *__restrict__ f, float *__restrict__ I) {
    constexpr int MAXC = 16;                                   // cells of a CTA at most
    __shared__ float2 tab[EXP2_N], K[MAXC][DIM + 5];                // u, -log2 e / (2 T), the four planes' factors
    __shared__ float B[MAXC];
    const int c0 = blockIdx.x * cells, nc = min(cells, n_cells - c0);
    if (threadIdx.x >= 32 && threadIdx.x < 32 + EXP2_N)
        tab[threadIdx.x - 32] = make_float2(g_exp2_table.hi[threadIdx.x - 32], g_exp2_table.lo[threadIdx.x - 32]);
    if (threadIdx.x < nc) {
        const double *M = F + (size_t)(c0 + threadIdx.x) * NF;
        auto put = [&](int k, double x) {
            const float h = (float)x;
            K[threadIdx.x][k] = make_float2(h, (float)(x - (double)h));
        };
        const double Tt = M[4];
        const double norm = M[0] * pow_neg_half_dim<DIM>(6.283185307179586 * Tt);
#pragma unroll
        for (int a = 0; a < DIM; ++a) put(a, M[1 + a]);
        put(DIM, -1.4426950408889634 / (2.0 * Tt));
        put(DIM + 1, norm);
        put(DIM + 2, (3 - DIM) * Tt * norm);
        put(DIM + 3, 0.5 * m.d_r * M[5] * norm);
        put(DIM + 4, vib_energy<double>(m, M[6]) * norm);
        B[threadIdx.x] = (float)(m.sigma_R * M[7] * M[7] * M[7] * M[7] / 3.141592653589793);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, nw = vq.n_pad / 32;
    for (int t = threadIdx.x >> 5; t < nc * nw; t += 8) {
        const int c = t / nw, v = (t - c * nw) * 32 + lane;
        float2 c2 = square2(two_diff(vq.x[v], K[c][0].x, K[c][0].y));
#pragma unroll
        for (int a = 1; a < DIM; ++a)
            c2 = add2w(c2, square2(two_diff(vq.x[a * vq.n_pad + v], K[c][a].x, K[c][a].y)));
        const Exp2 e = exp2_two(tab, K[c][DIM], c2);
        *reinterpret_cast<float4 *>(f + ((size_t)(c0 + c) * vq.n_pad + v) * 4) =
            make_float4(scaled(K[c][DIM + 1], e), DIM < 3 ? scaled(K[c][DIM + 2], e) : 0.0f, scaled(K[c][DIM + 3], e),
                        scaled(K[c][DIM + 4], e));
    }
    for (int t = threadIdx.x; t < nc * oq.n_pad; t += 256) I[(size_t)c0 * oq.n_pad + t] = B[t / oq.n_pad];
}

// ------------------------------------------------------------------ launchers
#define GSIS_DISPATCH_DIM(dim, ...)                    \
    switch (dim) {                                     \
        case 1: { constexpr int DIM = 1; __VA_ARGS__; } break; \
        case 2: { constexpr int DIM = 2; __VA_ARGS__; } break; \
        default: return cudaErrorInvalidValue;         \
    }
// the kinetic path (coefficients, wall density, slopes, sweeps, moments, finish,
// equilibrium) also runs on 3-D meshes
#define GSIS_DISPATCH_DIM3(dim, ...)                   \
    switch (dim) {                                     \
        case 1: { constexpr int DIM = 1; __VA_ARGS__; } break; \
        case 2: { constexpr int DIM = 2; __VA_ARGS__; } break; \
        case 3: { constexpr int DIM = 3; __VA_ARGS__; } break; \
        default: return cudaErrorInvalidValue;         \
    }

template <typename Real>
cudaError_t launch_coefficients(cudaStream_t s, int dim, const Geom<Real> &g, const ModelDev &m, const double *fields,
                                const double *cell_dx, Real *coef) {
    const int nt = 32, nbk = (g.n_cells + nt - 1) / nt;   // small CTAs spread the FP64 work over SMs
    GSIS_DISPATCH_DIM3(dim, (k_coefficients<Real, DIM><<<nbk, nt, 0, s>>>(g, m, fields, cell_dx, coef)));
    return cudaGetLastError();
}

template <typename Real>
cudaError_t launch_wall_density(cudaStream_t s, int dim, const Geom<Real> &g, const Quad<Real> &vq,
                                const double *patch_T, const double *bf_inc, const int *patch_kind, const Real *f,
                                const double *wout, Real *bcoef) {
    if (g.n_bf == 0) return cudaSuccess;
    GSIS_DISPATCH_DIM3(dim, (k_wall_density<Real, DIM><<<g.n_bf, 128, 0, s>>>(g, vq, patch_T, bf_inc, patch_kind, f,
                                                                             wout, bcoef)));
    return cudaGetLastError();
}

template <typename Real>
cudaError_t launch_wall_outflux(cudaStream_t s, int dim, const Geom<Real> &g, const Quad<Real> &vq,
                                const int *patch_kind, const Real *f, double *wout) {
    if (g.n_bf == 0) return cudaSuccess;
    GSIS_DISPATCH_DIM(dim, (k_wall_outflux<Real, DIM><<<g.n_bf, 128, 0, s>>>(g, vq, patch_kind, f, wout)));
    return cudaGetLastError();
}

// Per cell: the FP64 sums over the context's chunks of the gas and photon moment partials,
// X[cell][NXC] (gas moments first, photon moments at NMP): a velocity shard's share of
// every cell's moments, summed over the ranks and finished by launch_finish.
template <typename Real, int DIM>
__global__ void k_cell_sums(int n_cells, int n_chunks, int o_chunks, const Real *__restrict__ partial,
                            const Real *__restrict__ opartial, double *__restrict__ X) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_cells) return;
    constexpr int NM = n_gas_moments<DIM>();
    double S[NM];
    for (int k = 0; k < NM; ++k) S[k] = 0.0;
    for (int c = 0; c < n_chunks; ++c)
        for (int k = 0; k < NM; ++k) S[k] += (double)partial[((size_t)i * n_chunks + c) * NMP + k];
    double P[1 + DIM];
    for (int k = 0; k <= DIM; ++k) P[k] = 0.0;
    for (int c = 0; c < o_chunks; ++c)
        for (int k = 0; k <= DIM; ++k) P[k] += (double)opartial[((size_t)i * o_chunks + c) * NMO + k];
    double *x = X + (size_t)i * NXC;
    for (int k = 0; k < NXC; ++k) x[k] = 0.0;
    for (int k = 0; k < NM; ++k) x[k] = S[k];
    for (int k = 0; k <= DIM; ++k) x[NMP + k] = P[k];
}

template <typename Real>
cudaError_t launch_cell_sums(cudaStream_t s, int dim, int n_cells, int n_chunks, int o_chunks, const Real *partial,
                             const Real *opartial, double *X) {
    GSIS_DISPATCH_DIM(dim, (k_cell_sums<Real, DIM><<<(n_cells + 127) / 128, 128, 0, s>>>(n_cells, n_chunks, o_chunks,
                                                                                         partial, opartial, X)));
    return cudaGetLastError();
}

// Per cell: the rows of the synthetic equations (mass, momentum, total energy, e_r, e_v,
// e_R; stride NVM) of the moment partials of the kinetic residual that a sweep with
// Geom::resid leaves in partial / opartial.  The gas partials are about the velocity u0 of
// the cell's moment tile (coef of the tile's first cell, as the sweep took it):
//   sum xi r0 = sum c r0 + u0 sum r0,  sum |xi|^2 r0 = sum |c|^2 r0 + 2 u0 . sum c r0 + |u0|^2 sum r0.
template <typename Real, int DIM>
__global__ void k_resid_rows(int n_cells, int n_chunks, int o_chunks, const Real *__restrict__ coef,
                             const Real *__restrict__ partial, const Real *__restrict__ opartial,
                             double *__restrict__ rows) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_cells) return;
    constexpr int NM = n_gas_moments<DIM>(), NMPD = Lay<DIM>::NMP;
    double S[NM];
    for (int k = 0; k < NM; ++k) S[k] = 0.0;
    for (int c = 0; c < n_chunks; ++c)
        for (int k = 0; k < NM; ++k) S[k] += (double)partial[((size_t)i * n_chunks + c) * NMPD + k];
    double eR = 0.0;
    for (int c = 0; c < o_chunks; ++c) eR += (double)opartial[((size_t)i * o_chunks + c) * NMO];
    const Real *u = coef + (size_t)(i / MT * MT) * cf::NC + cf::U;
    double u0[DIM], uS = 0.0, u2 = 0.0, trc = 0.0;
    for (int a = 0; a < DIM; ++a) {
        u0[a] = (double)u[a];
        uS += u0[a] * S[1 + a];
        u2 += u0[a] * u0[a];
    }
    int m = 1 + DIM;
    for (int a = 0; a < DIM; ++a)
        for (int b = a; b < DIM; ++b, ++m)
            if (b == a) trc += S[m];
    m += DIM;                                  // past the c |c|^2 moments
    double plane[4] = {S[0], 0.0, 0.0, 0.0};   // sum r_p over the velocities
    for (int p = (DIM < 3 ? 1 : 2); p < 4; ++p) {
        plane[p] = S[m];
        m += 1 + DIM;
    }
    double *r = rows + (size_t)i * NVM;
    r[0] = S[0];
    for (int a = 0; a < DIM; ++a) r[1 + a] = S[1 + a] + u0[a] * S[0];
    r[1 + DIM] = 0.5 * (trc + 2.0 * uS + u2 * S[0]) + 0.5 * plane[1] + plane[2] + plane[3] + eR;
    r[2 + DIM] = plane[2];
    r[3 + DIM] = plane[3];
    r[4 + DIM] = eR;
}

template <typename Real>
cudaError_t launch_resid_rows(cudaStream_t s, int dim, int n_cells, int n_chunks, int o_chunks, const Real *coef,
                              const Real *partial, const Real *opartial, double *rows) {
    GSIS_DISPATCH_DIM3(dim, (k_resid_rows<Real, DIM><<<(n_cells + 127) / 128, 128, 0, s>>>(
                                n_cells, n_chunks, o_chunks, coef, partial, opartial, rows)));
    return cudaGetLastError();
}

template <typename Real, int N, int DIM>
static cudaError_t slopes_t(cudaStream_t s, const Geom<Real> &g, const Quad<Real> &q, const Real *f,
                            Real *fface) {
    if constexpr (std::is_same<Real, double>::value) {
        // few cells: one warp per CTA, so that the FP64 work reaches every SM
        const int cols = (q.n + 31) / 32, rows = (long long)g.n_cells * cols < SMS * SLOPE_ROWS ? 1 : SLOPE_ROWS;
        k_slopes64<N, DIM><<<dim3((g.n_cells + rows - 1) / rows, cols), dim3(32, rows), 0, s>>>(g, q.n, q.n_pad, q.x, f,
                                                                                             fface);
        return cudaGetLastError();
    } else {
        static_assert(SV % (32 * slope_vpt(DIM)) == 0, "a row's velocities must tile the padding");
        dim3 grid((g.n_cells + SLOPE_ROWS - 1) / SLOPE_ROWS, q.n_pad / (32 * slope_vpt(DIM))), block(32, SLOPE_ROWS);
        if (DIM < 3 && g.max_faces <= DIM + 1)     // segments, triangles
            k_slopes32<N, DIM, DIM + 1><<<grid, block, 0, s>>>(g, q.n, q.n_pad, q.x, f, fface);
        else
            k_slopes32<N, DIM, MAXF><<<grid, block, 0, s>>>(g, q.n, q.n_pad, q.x, f, fface);
        return cudaGetLastError();
    }
}

template <typename Real>
cudaError_t launch_slopes(cudaStream_t s, int dim, int planes, const Geom<Real> &g, const Quad<Real> &q,
                          const Real *f, Real *fface) {
    if (planes == 4) {
        GSIS_DISPATCH_DIM3(dim, return (slopes_t<Real, 4, DIM>(s, g, q, f, fface)));
    } else if (planes == 1) {
        GSIS_DISPATCH_DIM3(dim, return (slopes_t<Real, 1, DIM>(s, g, q, f, fface)));
    }
    return cudaErrorInvalidValue;
}

size_t sweep_smem_bytes(int block, int planes, int dim, size_t real_size, bool tc) {
    return sweep_main_bytes(block, planes, dim, real_size, tc) + (size_t)(dim + 1) * SV * real_size +
           (size_t)((block * MAXF + 15) & ~15) + (tc ? sizeof(tcm::Ctl) : 0);
}

// The dynamic shared memory a sweep may take: always the most a CTA can have, never this
// context's need.  The limit belongs to the kernel, and another thread's context, with another
// relaxation block, may set it between here and the launch.
template <typename K>
static cudaError_t allow_smem(K kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
}

template <typename Real, int N, int DIM, int ORDER, bool RESID>
static cudaError_t sweep_t(cudaStream_t s, const Geom<Real> &g, const Quad<Real> &q, const Real *coef,
                           const Real *bcoef, const Real *f_in, const Real *fface, Real *f_out, Real *partial) {
    const bool tc = N == 4 && sizeof(Real) == 4 && DIM < 3 && g.tc && !RESID;
    if (g.tc && (DIM == 3 || MT % g.block != 0)) return cudaErrorInvalidValue;
    dim3 grid((g.n_cells + g.block - 1) / g.block, q.n_pad / SV);
    auto run = [&](auto kern, dim3 block, size_t smem) {
        cudaError_t e = allow_smem(kern);
        if (e != cudaSuccess) return e;
        kern<<<grid, block, smem, s>>>(g, q, coef, bcoef, f_in, fface, f_out, partial);
        return cudaGetLastError();
    };
    const size_t smem = sweep_smem_bytes(g.block, N, DIM, sizeof(Real), tc);
    if constexpr (N == 4 && std::is_same<Real, float>::value) {
        if constexpr (DIM < 3 && !RESID)
            if (tc) return run(k_sweep<Real, N, DIM, ORDER>, dim3(SV, SROWS), smem);
        // segments and triangles, whose faces' values leave room for one more CTA per SM, or
        // any cells (the 20 000-triangle cavity as "any cells": 326 us, as triangles 306 us)
        const size_t bytes = S32<DIM>::bytes(g.block);
        if (g.block <= 2) return run(k_sweep_gas32<DIM, ORDER, RESID, MAXF, 1>, dim3(32), bytes);
        if (DIM < 3 && g.max_faces <= DIM + 1) return run(k_sweep_gas32<DIM, ORDER, RESID, DIM + 1, 4>, dim3(128), bytes);
        return run(k_sweep_gas32<DIM, ORDER, RESID, MAXF, 4>, dim3(128), bytes);
    } else {
        // FP64 on fewer (block, chunk) pairs than SMs: a pair's time is the FP64 pipe of the SM it
        // runs on.
        const long long pairs = (long long)grid.x * grid.y;
        if constexpr (N == 4) {
            // Gas: a cluster of eight CTAs per pair, while the chip holds all clusters at once (51,
            // 36 or 15 of them at three, two or one CTA per SM; a second wave costs as much as the
            // first) and the blocks have cells for the CTAs.  us of the 1-D sweep, cluster and one
            // CTA of eight rows: blocks of 16 cells 32 and 55 at 10 pairs, 45 and 55 at 50, 72 and
            // 55 at 57; of 32, 65 and 102 at 24, 118 and 102 at 38; of 64, 99 and 198 at 10, 193 and
            // 198 at 19, 383 and 198 at 50; of 8, 33 and 33 at 50; of 4, 21 and 22 at 10, 28 and 22
            // at 38; of 1, 18 and 16 at 10.
            const int per_sm = std::min<int>(3, 228 * 1024 / (smem + 1024));
            const int fit = per_sm == 3 ? 51 : per_sm == 2 ? 36 : 15;
            if (g.block >= 4 && pairs <= std::min(fit, 4 * g.block)) {
                auto kern = k_sweep<Real, N, DIM, ORDER, RESID, SROWS, 8>;
                cudaError_t e = allow_smem(kern);
                if (e != cudaSuccess) return e;
                cudaLaunchConfig_t cfg = {};
                cfg.gridDim = dim3(grid.x * 8, grid.y);
                cfg.blockDim = dim3(SV, SROWS);
                cfg.dynamicSmemBytes = smem;
                cfg.stream = s;
                cudaLaunchAttribute at = {};
                at.id = cudaLaunchAttributeClusterDimension;
                at.val.clusterDim.x = 8;
                at.val.clusterDim.y = at.val.clusterDim.z = 1;
                cfg.attrs = &at;
                cfg.numAttrs = 1;
                e = cudaLaunchKernelEx(&cfg, kern, g, q, coef, bcoef, f_in, fface, f_out, partial);
                return e != cudaSuccess ? e : cudaGetLastError();
            }
        }
        // one CTA of eight rows (blocks of 16 cells at 100 pairs: 55 us, of two rows 59); photons,
        // with few instructions per value, always
        if constexpr (std::is_same<Real, double>::value) {
            if (pairs < SMS) return run(k_sweep<Real, N, DIM, ORDER, RESID, 8>, dim3(SV, 8), smem);
        }
        return run(k_sweep<Real, N, DIM, ORDER, RESID>, dim3(SV, SROWS), smem);
    }
}

template <typename Real>
cudaError_t launch_sweep_gas(cudaStream_t s, int dim, int order, const Geom<Real> &g, const Quad<Real> &vq,
                             const Real *coef, const Real *bcoef, const Real *f_in, const Real *fface, Real *f_out,
                             Real *partial) {
    // g.resid selects the residual-only instantiation (the moments of the residual)
    if (order == 1 && g.resid) {
        GSIS_DISPATCH_DIM3(dim, return (sweep_t<Real, 4, DIM, 1, true>(s, g, vq, coef, bcoef, f_in, fface, f_out, partial)));
    } else if (order == 1) {
        GSIS_DISPATCH_DIM3(dim, return (sweep_t<Real, 4, DIM, 1, false>(s, g, vq, coef, bcoef, f_in, fface, f_out, partial)));
    } else if (g.resid) {
        GSIS_DISPATCH_DIM3(dim, return (sweep_t<Real, 4, DIM, 2, true>(s, g, vq, coef, bcoef, f_in, fface, f_out, partial)));
    } else {
        GSIS_DISPATCH_DIM3(dim, return (sweep_t<Real, 4, DIM, 2, false>(s, g, vq, coef, bcoef, f_in, fface, f_out, partial)));
    }
    return cudaErrorInvalidValue;
}

template <typename Real>
cudaError_t launch_sweep_photon(cudaStream_t s, int dim, int order, const Geom<Real> &g, const Quad<Real> &oq,
                                const Real *coef, const Real *bcoef, const Real *I_in, const Real *fface,
                                Real *I_out, Real *partial) {
    if (order == 1 && g.resid) {
        GSIS_DISPATCH_DIM3(dim, return (sweep_t<Real, 1, DIM, 1, true>(s, g, oq, coef, bcoef, I_in, fface, I_out, partial)));
    } else if (order == 1) {
        GSIS_DISPATCH_DIM3(dim, return (sweep_t<Real, 1, DIM, 1, false>(s, g, oq, coef, bcoef, I_in, fface, I_out, partial)));
    } else if (g.resid) {
        GSIS_DISPATCH_DIM3(dim, return (sweep_t<Real, 1, DIM, 2, true>(s, g, oq, coef, bcoef, I_in, fface, I_out, partial)));
    } else {
        GSIS_DISPATCH_DIM3(dim, return (sweep_t<Real, 1, DIM, 2, false>(s, g, oq, coef, bcoef, I_in, fface, I_out, partial)));
    }
    return cudaErrorInvalidValue;
}

template <typename Real>
cudaError_t launch_finish(cudaStream_t s, int dim, int n_cells, int n_chunks, int o_chunks, const ModelDev &m,
                          const Real *coef, const Real *partial, const Real *opartial, const double *vol,
                          const double *fields_old, double *fields_new, double *eps_terms, int *err_flag,
                          int have_old, double *eps_part, unsigned int *ticket, double *eps_sums,
                          const double *X) {
    const int nbk = (n_cells + 31) / 32, reduce = eps_sums != nullptr;
    auto go = [&](auto kern, int warps) {
        kern<<<nbk, 32 * warps, 0, s>>>(n_cells, n_chunks, o_chunks, m, coef, partial, opartial, vol, fields_old,
                                        fields_new, eps_terms, err_flag, have_old, reduce, eps_part, ticket, eps_sums,
                                        X);
    };
    if (n_chunks >= 4 && !X) GSIS_DISPATCH_DIM3(dim, go(k_finish<Real, DIM, 4>, 4))
    else GSIS_DISPATCH_DIM3(dim, go(k_finish<Real, DIM, 1>, 1))
    return cudaGetLastError();
}


template <typename Real>
cudaError_t launch_equilibrium(cudaStream_t s, int dim, int n_cells, const Quad<Real> &vq, const Quad<Real> &oq,
                               const ModelDev &m, const double *fields, Real *f, Real *I) {
    if constexpr (std::is_same<Real, float>::value) {
        // a cell's constants cost one thread about as much as 70 velocities cost a warp: 16 cells
        // to a CTA, fewer where that leaves SMs without one
        const int cells = std::max(1, std::min(16, n_cells / (2 * SMS))), grid = (n_cells + cells - 1) / cells;
        GSIS_DISPATCH_DIM3(dim, (k_equilibrium32<DIM><<<grid, 256, 0, s>>>(n_cells, cells, vq, oq, m, fields, f, I)));
    } else {
        GSIS_DISPATCH_DIM3(dim, (k_equilibrium<Real, DIM><<<n_cells, 256, 0, s>>>(n_cells, vq, oq, m, fields, f, I)));
    }
    return cudaGetLastError();
}

template <typename Real>
cudaError_t launch_moments_only(cudaStream_t s, int dim, int n_cells, bool tc, const Quad<Real> &vq,
                                const Quad<Real> &oq, const Real *coef, const Real *f, const Real *I, Real *partial, Real *opartial,
                                int tc_wait, int *err) {
    dim3 gg((n_cells + VCH / 32 - 1) / (VCH / 32), vq.n_pad / VCH);
    dim3 go((n_cells + 3) / 4, oq.n_pad / OCH);
    static_assert(VCH == tcm::K && SV == tcm::K, "moment chunks are the tensor-core K");
    bool on_tc = false;
    if constexpr (std::is_same<Real, float>::value) {
        if (tc && dim < 3) {     // the tensor-core basis covers the 1-D and 2-D moments
            const int nch = vq.n_pad / tcm::K, n_items = (n_cells + MT - 1) / MT * nch;
            GSIS_DISPATCH_DIM(dim, {
                auto kern = k_tc_pass<DIM, false>;
                kern<<<persistent_grid<DIM, false>(TC_SMEM, n_items), 128, TC_SMEM, s>>>(
                    n_cells, nch, n_items, vq, 0.f, nullptr, coef, const_cast<float *>(f), partial, tc_wait, err);
            });
            on_tc = true;
        }
    }
    if constexpr (std::is_same<Real, double>::value) {
        gg.x = (n_cells + VCH / 32 * MG - 1) / (VCH / 32 * MG);
        GSIS_DISPATCH_DIM3(dim, (k_moments_gas64<DIM><<<gg, VCH, 0, s>>>(n_cells, vq, coef, f, partial)));
    } else {
        if (!on_tc)
            GSIS_DISPATCH_DIM3(dim, (k_moments_gas<Real, DIM><<<gg, VCH, 0, s>>>(n_cells, vq, coef, f, partial)));
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    GSIS_DISPATCH_DIM3(dim, (k_moments_photon<Real, DIM><<<go, 128, 0, s>>>(n_cells, oq, I, opartial)));
    return cudaGetLastError();
}

template <typename Real>
cudaError_t launch_kinetic_bflux(cudaStream_t s, const MacroGeom &g, const ModelDev &m, const Quad<Real> &vq,
                                 const Quad<Real> &oq, const Real *f, const Real *I, double *kin_bflux, double *raw) {
    if (g.n_bf == 0) return cudaSuccess;
    if (raw && g.dim == 3) return cudaErrorInvalidValue;   // the shard exchange record holds 1-D/2-D sums
    GSIS_DISPATCH_DIM3(g.dim, (k_kinetic_bflux<Real, DIM><<<g.n_bf, 128, 0, s>>>(g, m, vq, oq, f, I, kin_bflux, raw)));
    return cudaGetLastError();
}

cudaError_t launch_kbflux_combine(cudaStream_t s, const MacroGeom &g, const double *raw, double *kin_bflux) {
    if (g.n_bf == 0) return cudaSuccess;
    GSIS_DISPATCH_DIM(g.dim, (k_kbflux_combine<DIM><<<(g.n_bf + 127) / 128, 128, 0, s>>>(g, raw, kin_bflux)));
    return cudaGetLastError();
}

template <typename Real>
cudaError_t launch_sync(cudaStream_t s, int dim, int n_cells, bool tc, const Quad<Real> &vq, const Quad<Real> &oq,
                        const ModelDev &m, double omega, const double *F_new, const double *F_half, const Real *coef,
                        Real *f, Real *I, Real *partial, Real *opartial, void *scratch, int tc_wait, int *err) {
    dim3 gg((n_cells + VCH / 32 - 1) / (VCH / 32), vq.n_pad / VCH);
    dim3 go((n_cells + 3) / 4, oq.n_pad / OCH);
    bool on_tc = false;
    if constexpr (std::is_same<Real, float>::value) {
        if (tc && dim < 3) {     // the tensor-core basis covers the 1-D and 2-D moments
            if (!scratch) return cudaErrorInvalidValue;
            float *kc = static_cast<float *>(scratch);
            const int nch = vq.n_pad / tcm::K, n_items = (n_cells + MT - 1) / MT * nch;
            const int smem = TC_SMEM + MT * SKC * (int)sizeof(float);
            GSIS_DISPATCH_DIM(dim, {
                k_sync_coef<DIM><<<(n_cells + 127) / 128, 128, 0, s>>>(n_cells, m, F_new, F_half, kc);
                auto kern = k_tc_pass<DIM, true>;
                kern<<<persistent_grid<DIM, true>(smem, n_items), 128, smem, s>>>(
                    n_cells, nch, n_items, vq, (float)omega, reinterpret_cast<const float4 *>(kc), coef, f, partial,
                    tc_wait, err);
            });
            on_tc = true;
        }
    }
    if (!on_tc)
        GSIS_DISPATCH_DIM3(dim, (k_sync_gas<Real, DIM><<<gg, VCH, 0, s>>>(n_cells, vq, m, omega, F_new, F_half, coef,
                                                                          f, partial)));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    GSIS_DISPATCH_DIM3(dim, (k_sync_photon<Real, DIM><<<go, 128, 0, s>>>(n_cells, oq, m, omega, F_new, F_half, I,
                                                                         opartial)));
    return cudaGetLastError();
}

#define GSIS_INSTANTIATE(Real)                                                                                     \
    template cudaError_t launch_coefficients<Real>(cudaStream_t, int, const Geom<Real> &, const ModelDev &,        \
                                                   const double *, const double *, Real *);                        \
    template cudaError_t launch_wall_density<Real>(cudaStream_t, int, const Geom<Real> &, const Quad<Real> &,     \
                                                   const double *, const double *, const int *, const Real *,      \
                                                   const double *, Real *);                                        \
    template cudaError_t launch_wall_outflux<Real>(cudaStream_t, int, const Geom<Real> &, const Quad<Real> &,     \
                                                   const int *, const Real *, double *);                           \
    template cudaError_t launch_cell_sums<Real>(cudaStream_t, int, int, int, int, const Real *, const Real *,      \
                                                double *);                                                         \
    template cudaError_t launch_resid_rows<Real>(cudaStream_t, int, int, int, int, const Real *, const Real *,     \
                                                 const Real *, double *);                                          \
    template cudaError_t launch_slopes<Real>(cudaStream_t, int, int, const Geom<Real> &, const Quad<Real> &,      \
                                             const Real *, Real *);                                                \
    template cudaError_t launch_sweep_gas<Real>(cudaStream_t, int, int, const Geom<Real> &, const Quad<Real> &,    \
                                                const Real *, const Real *, const Real *, const Real *, Real *,    \
                                                Real *);                                                           \
    template cudaError_t launch_sweep_photon<Real>(cudaStream_t, int, int, const Geom<Real> &, const Quad<Real> &, \
                                                   const Real *, const Real *, const Real *, const Real *, Real *, \
                                                   Real *);                                                        \
    template cudaError_t launch_finish<Real>(cudaStream_t, int, int, int, int, const ModelDev &, const Real *,     \
                                             const Real *, const Real *, const double *, const double *, double *, \
                                             double *, int *, int, double *, unsigned int *, double *,             \
                                             const double *);                                                      \
    template cudaError_t launch_equilibrium<Real>(cudaStream_t, int, int, const Quad<Real> &, const Quad<Real> &,  \
                                                  const ModelDev &, const double *, Real *, Real *);               \
    template cudaError_t launch_moments_only<Real>(cudaStream_t, int, int, bool, const Quad<Real> &,               \
                                                   const Quad<Real> &,                                             \
                                                   const Real *, const Real *, const Real *, Real *, Real *, int,  \
                                                   int *);                                                         \
    template cudaError_t launch_kinetic_bflux<Real>(cudaStream_t, const MacroGeom &, const ModelDev &,             \
                                                    const Quad<Real> &, const Quad<Real> &, const Real *,          \
                                                    const Real *, double *, double *);                             \
    template cudaError_t launch_sync<Real>(cudaStream_t, int, int, bool, const Quad<Real> &, const Quad<Real> &,   \
                                           const ModelDev &, double, const double *, const double *, const Real *, \
                                           Real *, Real *, Real *, Real *, void *, int, int *);

GSIS_INSTANTIATE(float)
GSIS_INSTANTIATE(double)

}  // namespace gsis
