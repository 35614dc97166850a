// Allocation-free velocity moments: gsis_moments_static.
//
// For callers that must not allocate device memory: code that runs while another
// component owns the device heap (a host framework with its own pool allocator, a
// plugin that may only use the buffers it is handed), or latency-critical loops that
// cannot afford a cudaMalloc/cudaFree pair per call.  Such callers cannot create a
// gsis context (gsis_create allocates), so this entry point takes device pointers.  It is
// one kernel (one of two) that keeps its intermediate sums in shared memory: calls share
// nothing, may overlap on a GPU and may be captured.
//
// Accuracy: the gas moments are summed about a per-cell shift velocity u0 (the cell's
// own mean velocity from a first pass over its mass and momentum), so that the third
// moments behind the heat fluxes do not cancel at high flow speeds; the FP32 storage
// path keeps 1e-5 of rho T^1.5 at Mach 5.  FP32 sums run over at most eight velocities per lane
// and are then carried in two words (Knuth's two-sum).
//
// What bounds it: the one pass over f (the second pass of a cell, right after the first,
// finds it in L1 or L2).  20 000 cells x 784 velocities, FP32: 301 -> 108 us (two passes over
// memory, an FP64 subtraction and conversion per velocity component and five kernels before).
// Few cells of large sets would leave most of the chip idle with a warp per cell: there a
// cluster of CTAs takes a cell (FP32, one cell of 9 216 velocities: 308 us by one warp, 19 by
// eight CTAs, 126 by the five kernels; FP64 389, 35 and 96).
#include <algorithm>
#include <cmath>
#include <cooperative_groups.h>
#include <type_traits>

#include "../../include/gsis.h"
#include "fp64.cuh"
#include "gsis_impl.cuh"

namespace {

using namespace gsis;

constexpr int kChunk = 128;                           // velocities (directions) counted as one by the size limit
constexpr int kNF = 26, kWarps = 8, kCpw = 4;         // record words; warps of a CTA; cells of a warp in a round
// 80 registers a thread: 2, 3, 4 CTAs per SM took 121, 102, 112 us on the case above
constexpr int kCtasPerSm = 3;
// bytes of the velocity sets in shared memory at most (three CTAs per SM hold 61 KB of them
// each, beside 14 KB of sums; between that and the limit two run)
constexpr int kMaxTable = 64 * 1024;
constexpr int kWideRun = 128;                         // velocities of a plain sum where a cell is split
// FP64: a cell is split among CTAs (k_static_wide) up to kWideCells cells, from kWideSet
// velocities or directions on.  us, split and whole: 64 x 784 22 and 74, 456 x 784 48 and 75,
// 700 x 784 74 and 75, 1 000 x 784 101 and 76, 700 x 9 216 484 and 738, 1 000 x 9 216 674 and
// 739; one cell of 9 216 35 and 389.
constexpr long long kWideCells = 700;
constexpr int kWideSet = 256;
constexpr int kRec = 24;                              // sums of a cell (gas, then photons), in threes

template <int DIM>
constexpr int n_moments() {
    return 1 + DIM + DIM * (DIM + 1) / 2 + DIM + 3 * (1 + DIM);
}

// The largest problem a call takes: the sums by chunks of 128 velocities or directions (20
// and 4 values in the storage type) and three doubles per cell come to at most 32 MiB.
// Callers may rely on larger ones being refused.
constexpr size_t kMaxBytes = size_t(32) << 20;
size_t problem_bytes(long long n_cells, int n_xi, int n_om, size_t real) {
    const size_t n_chunks = (n_xi + kChunk - 1) / kChunk, o_chunks = (n_om + kChunk - 1) / kChunk;
    return (size_t)n_cells * 3 * sizeof(double) + ((size_t)n_cells * n_chunks * 20 + (size_t)n_cells * o_chunks * 4) * real;
}

// A running sum: two words in FP32 (hi + lo, the rounding error of every addition kept), one
// in FP64
template <typename Real>
struct Sum;
template <>
struct Sum<float> {
    float hi = 0.0f, lo = 0.0f;
    __device__ __forceinline__ void add(float x) {
        const float t = hi + x, v = t - hi;
        lo += (hi - (t - v)) + (x - v);
        hi = t;
    }
    __device__ __forceinline__ void add(const Sum &o) {
        add(o.hi);
        lo += o.lo;
    }
    __device__ __forceinline__ Sum shfl(int o) const {
        Sum r;
        r.hi = __shfl_xor_sync(0xffffffffu, hi, o);
        r.lo = __shfl_xor_sync(0xffffffffu, lo, o);
        return r;
    }
    // an infinite hi leaves a NaN in lo
    __device__ __forceinline__ double value() const {
        return isfinite(lo) ? to_double(hi) + to_double(lo) : to_double(hi);
    }
};
template <>
struct Sum<double> {
    double hi = 0.0;
    __device__ __forceinline__ void add(double x) { hi += x; }
    __device__ __forceinline__ void add(const Sum &o) { hi += o.hi; }
    __device__ __forceinline__ Sum shfl(int o) const {
        Sum r;
        r.hi = __shfl_xor_sync(0xffffffffu, hi, o);
        return r;
    }
    __device__ __forceinline__ double value() const { return hi; }
};

// The velocity set as a lane reads it.  With a table in shared memory (FP32): each component in
// two floats, hi + lo, and the weight, converted once per CTA; else straight from the FP64 set.
template <typename Real, int DIM, bool TAB>
struct Velocities {
    const double *xi, *w;
    const float *tab;
    int n;
    __device__ __forceinline__ Real weight(int v) const {
        if constexpr (TAB) return tab[2 * DIM * n + v];
        else return to_real<Real>(w[v]);
    }
    // xi_a rounded (first pass)
    __device__ __forceinline__ Real x(int v, int a) const {
        if constexpr (TAB) return tab[a * n + v];
        else return to_real<Real>(xi[(size_t)v * DIM + a]);
    }
    // xi_a - u
    __device__ __forceinline__ Real minus(int v, int a, Real u) const {
        if constexpr (TAB) {
            return (tab[a * n + v] - u) + tab[(DIM + a) * n + v];
        } else {
            return to_real<Real>(xi[(size_t)v * DIM + a] - to_double(u));
        }
    }
};

// The photon directions likewise: weights and components in floats where TAB.
template <typename Real, int DIM, bool TAB>
struct Directions {
    const double *om, *wo;
    const float *tab;
    int n;
    __device__ __forceinline__ Real weight(int o) const {
        if constexpr (TAB) return tab[o];
        else return to_real<Real>(wo[o]);
    }
    __device__ __forceinline__ Real x(int o, int a) const {
        if constexpr (TAB) return tab[(1 + a) * n + o];
        else return to_real<Real>(om[(size_t)o * 3 + a]);
    }
};

// The four planes of a velocity; VEC: f is aligned to such a record, which is read at once
template <typename Real, bool VEC>
struct __align__((VEC ? 4 : 1) * sizeof(Real)) Planes {
    Real v[4];
};

// Mass and momentum of the velocities first, first + step, ... (a lane's), summed over the warp
template <int DIM, typename Real, typename Vel, typename Four>
__device__ __forceinline__ void mass_momentum(const Vel &vel, const Four *fc, int first, int step, int n_xi,
                                              Real (&m)[1 + DIM]) {
#pragma unroll
    for (int k = 0; k <= DIM; ++k) m[k] = Real(0);
#pragma unroll 8
    for (int v = first; v < n_xi; v += step) {
        const Real w0 = vel.weight(v) * fc[v].v[0];
        m[0] += w0;
#pragma unroll
        for (int a = 0; a < DIM; ++a) m[1 + a] += w0 * vel.x(v, a);
    }
#pragma unroll
    for (int k = 0; k <= DIM; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m[k] += __shfl_xor_sync(0xffffffffu, m[k], o);
}

// Adds a lane's share of the gas moments of the RUN velocities from v0 on, about u, to S
template <int DIM, int RUN, typename Real, typename Vel, typename Four>
__device__ __forceinline__ void add_gas_run(const Vel &vel, const Four *fc, int v0, int n_xi, int lane,
                                            const Real (&u)[DIM], Sum<Real> (&S)[kRec]) {
    constexpr int NM = n_moments<DIM>();
    Real acc[NM];
#pragma unroll
    for (int k = 0; k < NM; ++k) acc[k] = Real(0);
    // the run's loads first; past the set's end the last velocity again, which is not used
    Four fr[RUN / 32];
#pragma unroll
    for (int h = 0; h < RUN / 32; ++h) fr[h] = fc[min(v0 + 32 * h + lane, n_xi - 1)];
#pragma unroll
    for (int h = 0; h < RUN / 32; ++h) {
        const int v = v0 + 32 * h + lane;
        if (v >= n_xi) break;
        const Four &fv = fr[h];
        Real c[DIM], c2 = Real(0);
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            c[a] = vel.minus(v, a, u[a]);
            c2 = fma(c[a], c[a], c2);
        }
        const Real wv = vel.weight(v), w0 = wv * fv.v[0];
        Real wc[DIM];
        int k = 0;
        acc[k++] += w0;
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            wc[a] = w0 * c[a];
            acc[k++] += wc[a];
        }
#pragma unroll
        for (int a = 0; a < DIM; ++a)
#pragma unroll
            for (int b = a; b < DIM; ++b, ++k) acc[k] = fma(wc[a], c[b], acc[k]);
#pragma unroll
        for (int a = 0; a < DIM; ++a, ++k) acc[k] = fma(wc[a], c2, acc[k]);
#pragma unroll
        for (int p = 1; p < 4; ++p) {
            const Real wp = wv * fv.v[p];
            acc[k++] += wp;
#pragma unroll
            for (int a = 0; a < DIM; ++a, ++k) acc[k] = fma(wp, c[a], acc[k]);
        }
    }
#pragma unroll
    for (int k = 0; k < NM; ++k) S[k].add(acc[k]);
}

// the photon moments of the RUN directions from o0 on likewise
template <int DIM, int RUN, typename Real, typename Dir>
__device__ __forceinline__ void add_photon_run(const Dir &dir, const Real *Ic, int o0, int n_om, int lane,
                                               Sum<Real> (&S)[kRec]) {
    constexpr int NM = n_moments<DIM>();
    Real acc[1 + DIM];
#pragma unroll
    for (int k = 0; k <= DIM; ++k) acc[k] = Real(0);
#pragma unroll
    for (int h = 0; h < RUN / 32; ++h) {
        const int o = o0 + 32 * h + lane;
        if (o >= n_om) break;
        const Real wI = dir.weight(o) * Ic[o];
        acc[0] += wI;
#pragma unroll
        for (int a = 0; a < DIM; ++a) acc[1 + a] += wI * dir.x(o, a);
    }
#pragma unroll
    for (int k = 0; k <= DIM; ++k) S[NM + k].add(acc[k]);
}

// Sums S over the lanes: at the first three steps a lane passes half of its sums on, so that
// it ends with three, S[0..2], numbers first, first + 1, first + 2 (returned; the same in four
// consecutive lanes): 12 + 6 + 3 + 2 x 3 exchanges instead of 5 x 20
template <typename Real>
__device__ __forceinline__ int fold_lanes(int lane, Sum<Real> (&S)[kRec]) {
    int first = 0;
#pragma unroll
    for (int step = 0; step < 3; ++step) {
        const int half = 12 >> step, o = 16 >> step;
        const bool up = lane & o;
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            if (k >= half) break;
            const Sum<Real> a = S[k], b = S[half + k], got = (up ? a : b).shfl(o);
            S[k] = up ? b : a;
            S[k].add(got);
        }
        first += up ? half : 0;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        S[k].add(S[k].shfl(2));
        S[k].add(S[k].shfl(1));
    }
    return first;
}

// Sums S about u0 + the photon sums -> the cell's field record (rho, u, T_t, T_r, T_v, T_R,
// heat fluxes, stress).  u below is the residual velocity u - u0, and the central moments
// follow from it exactly as from moments about zero.
template <int DIM>
__device__ void finish(const double *S, const double *Ph, const double *u0, double i_half_dr, double i_half_dv,
                       double i_4sigma, double *F) {
    constexpr int MH = 3 - DIM;
    int k = 0;
    const double rho = S[k++], ir = rcp_r(rho);
    double m1[DIM], m2[DIM][DIM], m3[DIM];
    for (int a = 0; a < DIM; ++a) m1[a] = S[k++];
    for (int a = 0; a < DIM; ++a)
        for (int b = a; b < DIM; ++b) {
            m2[a][b] = m2[b][a] = S[k];
            ++k;
        }
    for (int a = 0; a < DIM; ++a) m3[a] = S[k++];
    const double H0 = S[k++];
    double Hc[DIM];
    for (int a = 0; a < DIM; ++a) Hc[a] = S[k++];
    const double G1 = S[k++];
    double G1c[DIM];
    for (int a = 0; a < DIM; ++a) G1c[a] = S[k++];
    const double G2 = S[k++];
    double G2c[DIM];
    for (int a = 0; a < DIM; ++a) G2c[a] = S[k++];
    double u[DIM], P[DIM][DIM], trP = 0.0, trm2 = 0.0, u2 = 0.0, um1 = 0.0;
    for (int a = 0; a < DIM; ++a) u[a] = m1[a] * ir;
    for (int a = 0; a < DIM; ++a)
        for (int b = 0; b < DIM; ++b) P[a][b] = m2[a][b] - rho * u[a] * u[b];
    for (int a = 0; a < DIM; ++a) {
        trP += P[a][a];
        trm2 += m2[a][a];
        u2 += u[a] * u[a];
        um1 += u[a] * m1[a];
    }
    const double ic2 = trP + H0;
    for (int q = 0; q < kNF; ++q) F[q] = 0.0;
    F[0] = rho;
    for (int a = 0; a < DIM; ++a) F[1 + a] = u0[a] + u[a];
    F[4] = ic2 * ((1.0 / 3.0) * ir);
    F[5] = G1 * (i_half_dr * ir);
    F[6] = G2 * (i_half_dv * ir);
    F[7] = i_4sigma > 0.0 ? sqrt_r(sqrt_r(fmax(Ph[0], 0.0) * i_4sigma)) : 0.0;
    for (int a = 0; a < DIM; ++a) {
        double t = m3[a] - u[a] * trm2 + u2 * m1[a] + 2.0 * u[a] * um1 - rho * u[a] * u2;
        for (int b = 0; b < DIM; ++b) t -= 2.0 * u[b] * m2[a][b];
        F[8 + a] = 0.5 * (t + Hc[a] - u[a] * H0);
        F[11 + a] = G1c[a] - u[a] * G1;
        F[14 + a] = G2c[a] - u[a] * G2;
        F[17 + a] = Ph[1 + a];
    }
    double sig[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    for (int a = 0; a < DIM; ++a)
        for (int b = 0; b < DIM; ++b) sig[a][b] = P[a][b];
    for (int a = DIM; a < 3; ++a) sig[a][a] = H0 * (1.0 / MH);
    for (int a = 0; a < 3; ++a) sig[a][a] -= ic2 * (1.0 / 3.0);
    F[20] = sig[0][0];
    F[21] = sig[1][1];
    F[22] = sig[2][2];
    F[23] = sig[0][1];
    F[24] = sig[0][2];
    F[25] = sig[1][2];
}

// One CTA takes a contiguous range of cells in rounds of 32, four per warp one after the
// other; one warp then forms the round's field records, one lane per cell (an FP64 warp
// instruction costs the same for one lane as for 32), while the others begin the next round
// in the second buffer.  VEC: f is aligned to a record of four planes, which is then read at once.
template <typename Real, int DIM, bool VEC>
__global__ void __launch_bounds__(32 * kWarps, kCtasPerSm) k_static(long long n_cells, int n_xi, int n_om,
                                                        const double *__restrict__ xi, const double *__restrict__ w,
                                                        const double *__restrict__ om, const double *__restrict__ wo,
                                                        const Real *__restrict__ f, const Real *__restrict__ I,
                                                        double i_half_dr, double i_half_dv, double i_4sigma, int per_cta,
                                                        double *__restrict__ out) {
    constexpr int NM = n_moments<DIM>();
    constexpr bool TAB = std::is_same<Real, float>::value;      // the FP32 sets are in shared memory
    constexpr int kRun = sizeof(Real) == 4 ? 256 : 128;   // velocities of a plain sum: 8 or 4 per lane, loaded at once
    static_assert(NM + 1 + DIM <= kRec && kWarps * kCpw == 32, "the sums of a cell; one lane per cell of a round");
    extern __shared__ float s_tab[];
    __shared__ double sums[2][kWarps * kCpw][kRec + 1], shift[2][kWarps * kCpw][DIM];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if constexpr (TAB) {
        for (int v = threadIdx.x; v < n_xi; v += 32 * kWarps) {
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                const double x = xi[(size_t)v * DIM + a];
                const float h = fp64::narrow(x);
                s_tab[a * n_xi + v] = h;
                s_tab[(DIM + a) * n_xi + v] = fp64::narrow(x - fp64::widen(h));
            }
            s_tab[2 * DIM * n_xi + v] = fp64::narrow(w[v]);
        }
        for (int o = threadIdx.x; o < n_om; o += 32 * kWarps) {
            float *q = s_tab + (2 * DIM + 1) * n_xi;
            q[o] = fp64::narrow(wo[o]);
#pragma unroll
            for (int a = 0; a < DIM; ++a) q[(1 + a) * n_om + o] = fp64::narrow(om[(size_t)o * 3 + a]);
        }
        __syncthreads();
    }
    const Velocities<Real, DIM, TAB> vel{xi, w, s_tab, n_xi};
    const float *pt = s_tab + (2 * DIM + 1) * n_xi;       // photon weights and directions
    const long long begin = (long long)blockIdx.x * per_cta, end = min(n_cells, begin + per_cta);
    const Directions<Real, DIM, TAB> dir{om, wo, pt, n_om};
    using Four = Planes<Real, VEC>;
    int round = 0;
    for (long long base = begin; base < end; base += kWarps * kCpw, ++round) {
        const int buf = round & 1;
        for (int j = 0; j < kCpw; ++j) {
            const int slot = j * kWarps + warp;
            const long long i = base + slot;
            if (i >= end) break;
            const Four *fc = reinterpret_cast<const Four *>(f) + (size_t)i * n_xi;
            // mass and momentum: the shift velocity (any value near the mean velocity serves)
            Real m[1 + DIM], u[DIM];
            mass_momentum<DIM>(vel, fc, lane, 32, n_xi, m);
#pragma unroll
            for (int a = 0; a < DIM; ++a) u[a] = m[0] > Real(0) ? m[1 + a] / m[0] : Real(0);
            Sum<Real> S[kRec];
            for (int v0 = 0; v0 < n_xi; v0 += kRun) add_gas_run<DIM, kRun>(vel, fc, v0, n_xi, lane, u, S);
            const Real *Ic = I + (size_t)i * n_om;
            for (int o0 = 0; o0 < n_om; o0 += kRun)
                add_photon_run<DIM, kRun>(dir, Ic, o0, n_om, lane, S);
            const int first = fold_lanes(lane, S);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const double x = S[k].value();
                if ((lane & 3) == 0) sums[buf][slot][first + k] = x;
            }
            if (lane == 0)
#pragma unroll
                for (int a = 0; a < DIM; ++a) shift[buf][slot][a] = to_double(u[a]);
        }
        __syncthreads();
        if (warp == round % kWarps && base + lane < end)
            finish<DIM>(sums[buf][lane], sums[buf][lane] + NM, shift[buf][lane], i_half_dr, i_half_dv, i_4sigma,
                        out + (size_t)(base + lane) * kNF);
    }
}

// One cell by a cluster of CTAs, whose warps take the cell's velocities in runs: for few cells,
// which k_static would leave to as many warps, and for FP32 sets too large for its tables (each
// component is then taken from the FP64 set).  The sums are added per warp, per CTA and over
// the cluster, each in a fixed order.
template <typename Real, int DIM, bool VEC>
__global__ void __launch_bounds__(32 * kWarps, kCtasPerSm) k_static_wide(int n_xi, int n_om, const double *__restrict__ xi,
                                                             const double *__restrict__ w,
                                                             const double *__restrict__ om,
                                                             const double *__restrict__ wo,
                                                             const Real *__restrict__ f, const Real *__restrict__ I,
                                                             double i_half_dr, double i_half_dv, double i_4sigma,
                                                             double *__restrict__ out) {
    constexpr int NM = n_moments<DIM>();
    __shared__ Real m_warp[kWarps][1 + DIM], m_cta[1 + DIM];
    __shared__ double sums[kRec], words[(kWarps + 1) * kRec];       // a Sum of either type is 8 bytes
    static_assert(sizeof(Sum<Real>) == sizeof(double), "sums in shared memory");
    Sum<Real> *s_warp = reinterpret_cast<Sum<Real> *>(words), *s_cta = s_warp + kWarps * kRec;
    const auto cluster = cooperative_groups::this_cluster();
    const int cs = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, wi = rank * kWarps + warp, nw = cs * kWarps;
    const size_t i = blockIdx.x / (unsigned)cs;
    using Four = Planes<Real, VEC>;
    const Four *fc = reinterpret_cast<const Four *>(f) + i * n_xi;
    const Velocities<Real, DIM, false> vel{xi, w, nullptr, n_xi};
    const Directions<Real, DIM, false> dir{om, wo, nullptr, n_om};
    Real m[1 + DIM], u[DIM];
    mass_momentum<DIM>(vel, fc, wi * 32 + lane, nw * 32, n_xi, m);
    if (lane == 0)
#pragma unroll
        for (int k = 0; k <= DIM; ++k) m_warp[warp][k] = m[k];
    __syncthreads();
    if (threadIdx.x <= DIM) {
        Real t = m_warp[0][threadIdx.x];
        for (int q = 1; q < kWarps; ++q) t += m_warp[q][threadIdx.x];
        m_cta[threadIdx.x] = t;
    }
    cluster.sync();
#pragma unroll
    for (int k = 0; k <= DIM; ++k) m[k] = Real(0);
    for (int r = 0; r < cs; ++r) {
        const Real *t = cluster.map_shared_rank(m_cta, r);
#pragma unroll
        for (int k = 0; k <= DIM; ++k) m[k] += t[k];
    }
#pragma unroll
    for (int a = 0; a < DIM; ++a) u[a] = m[0] > Real(0) ? m[1 + a] / m[0] : Real(0);
    Sum<Real> S[kRec];
    for (int v0 = wi * kWideRun; v0 < n_xi; v0 += nw * kWideRun)
        add_gas_run<DIM, kWideRun>(vel, fc, v0, n_xi, lane, u, S);
    for (int o0 = wi * kWideRun; o0 < n_om; o0 += nw * kWideRun)
        add_photon_run<DIM, kWideRun>(dir, I + i * n_om, o0, n_om, lane, S);
    const int first = fold_lanes(lane, S);
    if ((lane & 3) == 0)
#pragma unroll
        for (int k = 0; k < 3; ++k) s_warp[warp * kRec + first + k] = S[k];
    __syncthreads();
    if (threadIdx.x < kRec) {
        Sum<Real> t = s_warp[threadIdx.x];
        for (int q = 1; q < kWarps; ++q) t.add(s_warp[q * kRec + threadIdx.x]);
        s_cta[threadIdx.x] = t;
    }
    cluster.sync();
    if (rank == 0 && threadIdx.x < kRec) {
        Sum<Real> t = s_cta[threadIdx.x];
        for (int r = 1; r < cs; ++r) t.add(cluster.map_shared_rank(s_cta, r)[threadIdx.x]);
        sums[threadIdx.x] = t.value();
    }
    cluster.sync();      // the other CTAs' shared memory has been read
    if (rank == 0 && threadIdx.x == 0) {
        double u0[DIM];
#pragma unroll
        for (int a = 0; a < DIM; ++a) u0[a] = to_double(u[a]);
        finish<DIM>(sums, sums + NM, u0, i_half_dr, i_half_dv, i_4sigma, out + i * kNF);
    }
}

template <typename Real, int DIM>
int run(long long n_cells, int n_xi, const double *xi, const double *w, int n_om, const double *om,
        const double *wo, const void *f, const void *I, double d_r, double d_v, double sigma_R, double *out,
        cudaStream_t s) {
    if (problem_bytes(n_cells, n_xi, n_om, sizeof(Real)) > kMaxBytes) return GSIS_ERR_INVALID_ARG;
    // kCtasPerSm CTAs per SM share the cells out evenly; few cells: one per warp
    constexpr int slots = SMS * kCtasPerSm;
    const long long per = std::max<long long>(kWarps, (n_cells + slots - 1) / slots);
    const unsigned ctas = (unsigned)((n_cells + per - 1) / per);
    auto go = [&](auto kern, size_t smem) {
        // always the bound, never this call's size: the limit belongs to the kernel, and another
        // thread's call may set it between here and the launch
        if (smem > 16384 &&
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxTable) != cudaSuccess)
            return GSIS_ERR_CUDA;
        kern<<<ctas, 32 * kWarps, smem, s>>>(n_cells, n_xi, n_om, xi, w, om, wo, static_cast<const Real *>(f),
                                             static_cast<const Real *>(I), 2.0 / d_r, 2.0 / d_v,
                                             sigma_R > 0.0 ? 1.0 / (4.0 * sigma_R) : 0.0, (int)per, out);
        return cudaGetLastError() == cudaSuccess ? GSIS_OK : GSIS_ERR_CUDA;
    };
    const bool vec = reinterpret_cast<uintptr_t>(f) % (4 * sizeof(Real)) == 0;
    auto go_wide = [&](auto kern) {
        // as many CTAs per cell as give every warp a run and leave no SM without work
        int cs = 1;
        while (cs < 8 && n_cells * cs <= SMS && std::max(n_xi, n_om) > cs * kWarps * kWideRun) cs *= 2;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(n_cells * cs));
        cfg.blockDim = dim3(32 * kWarps);
        cfg.stream = s;
        cudaLaunchAttribute at = {};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = cs;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, n_xi, n_om, xi, w, om, wo, static_cast<const Real *>(f),
                                                 static_cast<const Real *>(I), 2.0 / d_r, 2.0 / d_v,
                                                 sigma_R > 0.0 ? 1.0 / (4.0 * sigma_R) : 0.0, out);
        return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? GSIS_OK : GSIS_ERR_CUDA;
    };
    // FP32: the tables of the sets while they fit (4 000 cells x 2 304 velocities with them 99 us,
    // one cell 23); beyond, split, with or without few cells (4 096 velocities, one cell 15 us and
    // 131 unsplit, 1 000 cells 86 and 156, 4 000 cells 294 and 441)
    const size_t tab = ((size_t)n_xi * (2 * DIM + 1) + (size_t)n_om * (1 + DIM)) * sizeof(float);
    constexpr bool fp32 = std::is_same<Real, float>::value;
    if (fp32 ? tab > kMaxTable : n_cells <= kWideCells && std::max(n_xi, n_om) >= kWideSet)
        return vec ? go_wide(k_static_wide<Real, DIM, true>) : go_wide(k_static_wide<Real, DIM, false>);
    return vec ? go(k_static<Real, DIM, true>, fp32 ? tab : 0) : go(k_static<Real, DIM, false>, fp32 ? tab : 0);
}

}  // namespace

extern "C" int gsis_moments_static(int32_t dim, int32_t precision, int64_t n_cells, int32_t n_xi, const double *xi,
                                   const double *w, int32_t n_omega, const double *omega, const double *wo,
                                   const void *f, const void *I, double d_r, double d_v, double sigma_R,
                                   double *fields, void *cuda_stream) {
    if (n_cells <= 0 || n_xi <= 0 || n_omega <= 0 || !xi || !w || !omega || !wo || !f || !I || !fields)
        return GSIS_ERR_INVALID_ARG;
    if (!(d_r > 0) || !(d_v > 0) || !(sigma_R >= 0)) return GSIS_ERR_INVALID_ARG;
    if (n_cells > (1LL << 31) / 4) return GSIS_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    if (dim == 3) return GSIS_ERR_UNSUPPORTED;
    if (dim != 1 && dim != 2) return GSIS_ERR_INVALID_ARG;
    if (precision == GSIS_FP32)
        return dim == 1 ? run<float, 1>(n_cells, n_xi, xi, w, n_omega, omega, wo, f, I, d_r, d_v, sigma_R, fields, s)
                        : run<float, 2>(n_cells, n_xi, xi, w, n_omega, omega, wo, f, I, d_r, d_v, sigma_R, fields, s);
    if (precision == GSIS_FP64)
        return dim == 1 ? run<double, 1>(n_cells, n_xi, xi, w, n_omega, omega, wo, f, I, d_r, d_v, sigma_R, fields, s)
                        : run<double, 2>(n_cells, n_xi, xi, w, n_omega, omega, wo, f, I, d_r, d_v, sigma_R, fields, s);
    return GSIS_ERR_INVALID_ARG;
}
