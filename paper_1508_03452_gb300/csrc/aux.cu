// aux.cu -- initial state, open boundaries, normal-B fix, photospheric driving,
// output conversion and float64 diagnostics of the RRMHD lattice Boltzmann
// library (arXiv:1508.03452, Secs. III-IV).
#include <math_constants.h>

#include <climits>
#include <cstddef>
#include <cstring>

#include "aux.cuh"
#include "pair.cuh"

namespace lb {

// ---------------------------------------------------------------------------
// helpers
// ---------------------------------------------------------------------------
template <class Cfg>
__device__ __forceinline__ void load_prim(const typename Cfg::prim* P, int64_t stride, int64_t c,
                                          Prim<typename Cfg::real>& s)
{
    using R = typename Cfg::real;
    s.n = (R)P[prim_elem(P_N, c, stride)];
    s.eps = (R)P[prim_elem(P_EPS, c, stride)];
    for (int a = 0; a < 3; ++a) {
        s.u[a] = (R)P[prim_elem(P_U + a, c, stride)];
        s.E[a] = (R)P[prim_elem(P_E + a, c, stride)];
        s.B[a] = (R)P[prim_elem(P_B + a, c, stride)];
    }
    s.rho = (R)P[prim_elem(P_RHO, c, stride)];
}

template <class Cfg, class R>
__device__ __forceinline__ void store_prim(typename Cfg::prim* P, int64_t stride, int64_t c, const Prim<R>& s)
{
    using T = typename Cfg::prim;
    P[prim_elem(P_N, c, stride)] = (T)s.n;
    P[prim_elem(P_EPS, c, stride)] = (T)s.eps;
    for (int a = 0; a < 3; ++a) {
        P[prim_elem(P_U + a, c, stride)] = (T)s.u[a];
        P[prim_elem(P_E + a, c, stride)] = (T)s.E[a];
        P[prim_elem(P_B + a, c, stride)] = (T)s.B[a];
    }
    P[prim_elem(P_RHO, c, stride)] = (T)s.rho;
}

template <int I, class Cfg, class R>
struct EqStore {
    static __device__ __forceinline__ void run(const PopView<Cfg>& V, int64_t c, const EqCell<R>& q)
    {
        st_pop<Cfg>(V.fg + fg_elem(I, 0, c, V.stride), (typename Cfg::real)feq_dev<I>(q), V.hs.finv[I]);
        st_pop<Cfg>(V.fg + fg_elem(I, 1, c, V.stride), (typename Cfg::real)geq_dev<I>(q), V.hs.ginv[I]);
        EqStore<I + 1, Cfg, R>::run(V, c, q);
    }
};
template <class Cfg, class R>
struct EqStore<19, Cfg, R> {
    static __device__ __forceinline__ void run(const PopView<Cfg>&, int64_t, const EqCell<R>&) {}
};

template <int K, class Cfg, class R>
struct HeqStore {
    static __device__ __forceinline__ void run(const PopView<Cfg>& V, int64_t c, const R* E, const R* B, const R* J,
                                               const Phys<R>& k)
    {
        V.h[h_elem(K, c, V.stride)] = (typename Cfg::hpop)heq13<K>(E, B, J, k);
        HeqStore<K + 1, Cfg, R>::run(V, c, E, B, J, k);
    }
};
template <class Cfg, class R>
struct HeqStore<24, Cfg, R> {
    static __device__ __forceinline__ void run(const PopView<Cfg>&, int64_t, const R*, const R*, const R*,
                                               const Phys<R>&) {}
};

// Conversions between float32 and float64 on the integer pipes, the same values as
// the conversion instructions (which flush subnormal float32, -ftz=true): those share
// GB300's float64 pipe (two lanes per SM), which bounds the passes below. All cases in
// integers: an instruction in a rare branch is executed for every value, the compiler
// turns the branch into a selection.
__device__ __forceinline__ double widen(float v)
{
    const unsigned u = __float_as_uint(v), m = u & 0x7fffffffu;
    const unsigned hi = (m >> 3) + (m >= 0x7f800000u ? 0x70000000u : 0x38000000u);  // (infinity, NaN: all exponent bits)
    const bool zero = m < 0x00800000u;
    return __hiloint2double((int)((u & 0x80000000u) | (zero ? 0u : hi)), zero ? 0 : (int)(u << 29));
}
__device__ __forceinline__ double widen(double v) { return v; }

template <class T>
__device__ __forceinline__ T narrow(double v);
template <>
__device__ __forceinline__ double narrow<double>(double v)
{
    return v;
}
template <>
__device__ __forceinline__ float narrow<float>(double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned hi = (unsigned)(b >> 32), m = hi & 0x7fffffffu;
    // a normal float32: round to nearest even at bit 29 (up to infinity), move the exponent
    const unsigned long long r = b + 0x0fffffffull + ((b >> 29) & 1ull);
    unsigned o = ((unsigned)(r >> 29) - 0xc0000000u) & 0x7fffffffu;
    o = m < 0x38100000u ? 0u : o;           // below 2^-126
    o = m >= 0x47f00000u ? 0x7f800000u : o;  // from 2^128 on, infinity
    o = m > 0x7ff00000u || (m == 0x7ff00000u && (unsigned)b != 0u) ? 0x7fffffffu : o;  // NaN
    return __uint_as_float((hi & 0x80000000u) | o);
}

template <class T>
__device__ __forceinline__ T narrow(FloatPair v)  // (float32 storage only)
{
    return (T)v.h;
}
// the type the initial state's equilibria are formed in: float64, or float32 pairs
// where the results are stored as float32 (and float16). 48 bits are enough for sums
// and products of deviations, not for what cancels to one: those are float64 in both
// (set_equilibrium_init). The populations then are float64's deviations rounded to
// float32, but for the rare value whose 48 bits do not settle the rounding.
template <class Cfg>
struct InitReal {
    using type = FloatPair;
};
template <>
struct InitReal<CfgF64> {
    using type = double;
};
template <class Q>
__device__ __forceinline__ Q split(double v);
template <>
__device__ __forceinline__ double split<double>(double v)
{
    return v;
}
template <>
__device__ __forceinline__ FloatPair split<FloatPair>(double v)
{
    const float h = narrow<float>(v);
    return {h, narrow<float>(v - widen(h))};
}
inline const Phys<double>& init_phys(const Phys<double>& k, double) { return k; }
inline Phys<FloatPair> init_phys(const Phys<double>& k, FloatPair) { return pair_phys(k); }

// post-equilibrium f and g of the opposite directions of group G from terms of type Q
template <int G, class Cfg, class Q>
struct EqStoreEven {
    static __device__ __forceinline__ void run(const PopView<Cfg>& V, int64_t c, const EqEvenT<Q>& e)
    {
        using R = typename Cfg::real;
        if constexpr (G == 0) {
            st_fgpair<Cfg>(V.fg + fg_elem(0, 0, c, V.stride), narrow<R>(e.f0), narrow<R>(e.g0), V.hs.finv[0], V.hs.ginv[0]);
        } else {
            constexpr int I = 2 * G - 1, a = ax1(I), b = ax2(I);
            static_assert(c19(I, a) == 1, "the first direction of a group points along its first axis");
            Q fe, fo, ge, go;
            if constexpr (b < 0) {
                fe = e.fe_ax[a], fo = e.fo_ax[a], ge = e.ge_ax[a], go = e.go_ax[a];
            } else {
                constexpr int m = a + b - 1;
                constexpr bool plus = c19(I, b) > 0;
                fe = plus ? e.fe_dg[m] + e.fx[m] : e.fe_dg[m] - e.fx[m];
                fo = plus ? e.fo_dg[a] + e.fo_dg[b] : e.fo_dg[a] - e.fo_dg[b];
                ge = plus ? e.ge_dg[m] + e.gx[m] : e.ge_dg[m] - e.gx[m];
                go = plus ? e.go_dg[a] + e.go_dg[b] : e.go_dg[a] - e.go_dg[b];
            }
            st_quad<Cfg>(V.fg + fg_elem(I, 0, c, V.stride),
                         V4<R>{narrow<R>(fe + fo), narrow<R>(ge + go), narrow<R>(fe - fo), narrow<R>(ge - go)},
                         V4<float>{V.hs.finv[I], V.hs.ginv[I], V.hs.finv[I + 1], V.hs.ginv[I + 1]});
        }
        EqStoreEven<G + 1, Cfg, Q>::run(V, c, e);
    }
};
template <class Cfg, class Q>
struct EqStoreEven<kFGroups + 1, Cfg, Q> {
    static __device__ __forceinline__ void run(const PopView<Cfg>&, int64_t, const EqEvenT<Q>&) {}
};

// h^eq of plane P's pairs: a +- (e - m), a and e being +-(sum or difference) of the two
// scaled components of J and E
template <int P, class Cfg, class Q>
__device__ __forceinline__ void heq_store_plane(const PopView<Cfg>& V, int64_t c, const Q* E, const Q* B, const Q* J,
                                                const Phys<Q>& k)
{
    constexpr int a1 = plane_a1(P), a2 = plane_a2(P);
    const Q js = Q(kSqrt2 / 16.0) * k.c, es = Q(kSqrt2 / 16.0) * k.inv_c;
    const Q j1 = js * J[a1], j2 = js * J[a2], e1 = es * E[a1], e2 = es * E[a2];
    const Q m = Q(0.125 * plane_orient(P)) * B[plane_normal(P)];
    const Q jp = j1 + j2, jm = j1 - j2, ep = e1 + e2, em = e1 - e2;
    // hops (+,+), (-,+), (-,-), (+,-); the e of pair i lies along hop i - 1
    const Q a[4] = {jp, -jm, -jp, jm}, x[4] = {em - m, ep - m, -em - m, -ep - m};
#pragma unroll
    for (int i = 0; i < 4; ++i)
        st_hpair<Cfg>(V.h + h_elem(8 * P + 2 * i, c, V.stride), narrow<typename Cfg::real>(a[i] + x[i]),
                      narrow<typename Cfg::real>(a[i] - x[i]));
}

// J from Eq. Ohm, g the Lorentz factor; F = E + u x B and Eu = E.u / c^2, of which F
// cancels in an ideal state and Eu across the flow
__device__ __forceinline__ void ohm_terms(const double* E, const double* u, const double* B, double inv_c2, double* F,
                                          double& Eu)
{
    Eu = (E[0] * u[0] + E[1] * u[1] + E[2] * u[2]) * inv_c2;
    F[0] = fma(u[1], B[2], fma(-u[2], B[1], E[0]));
    F[1] = fma(u[2], B[0], fma(-u[0], B[2], E[1]));
    F[2] = fma(u[0], B[1], fma(-u[1], B[0], E[2]));
}
template <class Q>
__device__ __forceinline__ void ohm_current_terms(const Q* F, Q Eu, const Q* u, Q rho, Q g, const Phys<Q>& k, Q* J)
{
    const Q sg = k.sigma * g;
    for (int a = 0; a < 3; ++a) J[a] = fma(rho, u[a], sg * fma(-Eu, u[a], F[a]));
}
__device__ __forceinline__ void ohm_current_g(const double* E, const double* u, const double* B, double rho, double g,
                                              const Phys<double>& k, double* J)
{
    double F[3], Eu;
    ohm_terms(E, u, B, k.inv_c * k.inv_c, F, Eu);
    ohm_current_terms(F, Eu, u, rho, g, k, J);
}

// the constants of a run that the initial state's float64 differences take
struct InitPhys {
    double c2, inv_c2, gm1, inv_gm1, eps0_2dx, n_r, eps_r, Er[3], Br[3];
};
inline InitPhys init_consts(const Phys<double>& k)
{
    return {k.c2,    k.inv_c * k.inv_c, k.gm1, 1.0 / k.gm1, k.eps0 / (2.0 * k.dx), k.n_r, k.eps_r, {k.Er[0], k.Er[1], k.Er[2]},
            {k.Br[0], k.Br[1], k.Br[2]}};
}

// Every population of cell c at its equilibrium for primitives s. The deviations from
// the reference state, the pressure's, 1 - u^2 / c^2 and Ohm's E + u x B are
// differences of near-equal numbers: float64, and only then of type Q. (With the
// differences taken in float32 pairs a deviation of relative size d was wrong by
// ~2e-15 / d of itself, and J of an ideal state by ~2e-15 sigma |u| |B|.)
template <class Cfg, class Q>
__device__ __forceinline__ void set_equilibrium_init(const PopView<Cfg>& V, int64_t c, const Prim<double>& s,
                                                     const InitPhys& w, const Phys<Q>& k)
{
    const double n_dev = s.n - w.n_r, eps_dev = s.eps - w.eps_r;
    const Q p_dev = split<Q>(w.gm1 * (eps_dev - n_dev * w.c2));
    const double b2 = (s.u[0] * s.u[0] + s.u[1] * s.u[1] + s.u[2] * s.u[2]) * w.inv_c2;
    Lorentz<Q> lz;
    lz.g = rsqrt_newton(split<Q>(1.0 - b2));
    lz.g2 = lz.g * lz.g;
    lz.gm1 = lz.g2 * split<Q>(b2) * rcp_approx(lz.g + Q(1));
    double F[3], Eu;
    ohm_terms(s.E, s.u, s.B, w.inv_c2, F, Eu);
    Prim<Q> q;
    q.n = split<Q>(s.n);
    q.eps = split<Q>(s.eps);
    q.rho = split<Q>(s.rho);
    Q J[3], Fq[3], dE[3], dB[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        q.u[a] = split<Q>(s.u[a]);
        q.E[a] = split<Q>(s.E[a]);
        q.B[a] = split<Q>(s.B[a]);
        Fq[a] = split<Q>(F[a]);
        dE[a] = split<Q>(s.E[a] - w.Er[a]);
        dB[a] = split<Q>(s.B[a] - w.Br[a]);
    }
    ohm_current_terms(Fq, split<Q>(Eu), q.u, q.rho, lz.g, k, J);
    heq_store_plane<0, Cfg>(V, c, dE, dB, J, k);
    heq_store_plane<1, Cfg>(V, c, dE, dB, J, k);
    heq_store_plane<2, Cfg>(V, c, dE, dB, J, k);
    EqCell<Q> eq;
    eq_cell(q, split<Q>(n_dev), split<Q>(eps_dev), dE, dB, k, eq, &lz, &p_dev);
    EqEvenT<Q> e;
    eq_even(eq, e);
    EqStoreEven<0, Cfg, Q>::run(V, c, e);
}

// every population of cell c at its equilibrium for primitives s (the
// post-collision value of an equilibrium state is the equilibrium itself)
template <class Cfg, class R>
__device__ __forceinline__ void set_equilibrium(const PopView<Cfg>& V, int64_t c, const Prim<R>& s, const Phys<R>& k)
{
    EqCell<R> q;
    eq_cell(s, k, q);
    R J[3];
    ohm_current(s.E, s.u, s.B, s.rho, k, J);
    EqStore<0, Cfg, R>::run(V, c, q);
    const R dE[3] = {s.E[0] - k.Er[0], s.E[1] - k.Er[1], s.E[2] - k.Er[2]};
    const R dB[3] = {s.B[0] - k.Br[0], s.B[1] - k.Br[1], s.B[2] - k.Br[2]};
    HeqStore<0, Cfg, R>::run(V, c, dE, dB, J, k);
    V.h[h_elem(24, c, V.stride)] = (typename Cfg::hpop)s.rho;
}

// ---------------------------------------------------------------------------
// initial state (Sec. IV set-ups): eps from Eq. EOS, E = -u x B when not
// given (Eq. Ohm_ideal), rho_c = eps0 div E by central differences (Eq.
// Gauss_E), J from Eq. Ohm, populations at equilibrium. float64 arithmetic.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void input_E(const InitInputs& in, int64_t c, int64_t N, double* E)
{
    if (in.E) {
        E[0] = in.E[c]; E[1] = in.E[N + c]; E[2] = in.E[2 * N + c];
    } else {
        const double u[3] = {in.u[c], in.u[N + c], in.u[2 * N + c]};
        const double B[3] = {in.B[c], in.B[N + c], in.B[2 * N + c]};
        E[0] = -(u[1] * B[2] - u[2] * B[1]);
        E[1] = -(u[2] * B[0] - u[0] * B[2]);
        E[2] = -(u[0] * B[1] - u[1] * B[0]);
    }
}

// component A of the input E at cell c
template <int A>
__device__ __forceinline__ double input_E1(const InitInputs& in, int64_t c, int64_t N)
{
    if (in.E) return in.E[A * N + c];
    constexpr int p = (A + 1) % 3, q = (A + 2) % 3;
    return -(in.u[p * N + c] * in.B[q * N + c] - in.u[q * N + c] * in.B[p * N + c]);
}

// Bound by arithmetic, in float64 by GB300's rate of two lanes per SM: opposite
// directions share the even and odd parts of their equilibria, a plane's Maxwell pairs
// their sums, one Lorentz factor serves J and the equilibria, and where the results
// are stored in float32 all but E, div E and what cancels is in float32 pairs. 256^3
// cells in float32: 21.5 ms direction by direction in float64, 14.3 with the terms
// shared, 4.9 with the pairs (memory would take 0.9; 9.3 with the conversions' rare cases
// left to the instructions).
template <class Cfg>
__global__ void __launch_bounds__(128) init_kernel(PopView<Cfg> V, InitInputs in, Phys<typename InitReal<Cfg>::type> k,
                                                   InitPhys w, int* bad)
{
    const int64_t N = (int64_t)V.nx * V.ny * V.nz;
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c >= N) return;
    const int x = (int)(c % V.nx), y = (int)((c / V.nx) % V.ny), z = (int)(c / ((int64_t)V.nx * V.ny));
    Prim<double> s;
    s.n = in.n[c];
    // p / (Gamma - 1): the product with the reciprocal, corrected by its remainder (as the
    // division rounds; an infinite p has no remainder)
    const double p = in.p[c], pq = p * w.inv_gm1;
    const bool over = ((unsigned)__double2hiint(pq) & 0x7ff00000u) == 0x7ff00000u;
    s.eps = s.n * w.c2 + (over ? pq : fma(fma(-pq, w.gm1, p), w.inv_gm1, pq));
    for (int a = 0; a < 3; ++a) {
        s.u[a] = in.u[a * N + c];
        s.B[a] = in.B[a * N + c];
    }
    input_E(in, c, N, s.E);
    if (!(s.u[0] * s.u[0] + s.u[1] * s.u[1] + s.u[2] * s.u[2] < w.c2) || !(s.n > 0)) atomicExch(bad, 1);
    // rho_c = eps0 div E
    double div = 0.0;
    if (V.nx > 1) {
        const int64_t row = c - x;
        div += input_E1<0>(in, row + wrap_coord(x + 1, V.nx, V.periodic[0]), N) -
               input_E1<0>(in, row + wrap_coord(x - 1, V.nx, V.periodic[0]), N);
    }
    if (V.ny > 1) {
        const int64_t col = c - (int64_t)V.nx * y;
        div += input_E1<1>(in, col + (int64_t)V.nx * wrap_coord(y + 1, V.ny, V.periodic[1]), N) -
               input_E1<1>(in, col + (int64_t)V.nx * wrap_coord(y - 1, V.ny, V.periodic[1]), N);
    }
    if (V.nz > 1) {
        const int64_t plane = (int64_t)V.nx * V.ny, col = c - plane * z;
        div += input_E1<2>(in, col + plane * wrap_coord(z + 1, V.nz, V.periodic[2]), N) -
               input_E1<2>(in, col + plane * wrap_coord(z - 1, V.nz, V.periodic[2]), N);
    }
    s.rho = w.eps0_2dx * div;
    {
        typename Cfg::prim pv[NPRIM];
        pv[P_N] = narrow<typename Cfg::prim>(s.n);
        pv[P_EPS] = narrow<typename Cfg::prim>(s.eps);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            pv[P_U + a] = narrow<typename Cfg::prim>(s.u[a]);
            pv[P_E + a] = narrow<typename Cfg::prim>(s.E[a]);
            pv[P_B + a] = narrow<typename Cfg::prim>(s.B[a]);
        }
        pv[P_RHO] = narrow<typename Cfg::prim>(s.rho);
        st_prims<Cfg>(V.prim + prim_elem(0, c, V.stride), V.stride, pv);
    }
    V.h[h_elem(24, c, V.stride)] = narrow<typename Cfg::hpop>(s.rho);
    set_equilibrium_init<Cfg>(V, c, s, w, k);
}

// float64 means for the reference state: n, p, E (3), B (3), E_a E_b (6: xx yy
// zz xy xz yz), B_a B_b (6), B x E (3). Pass 1: per-block partial sums
// (grid-stride); pass 2: one block adds the partials in block order, so the
// result does not depend on scheduling.
__global__ void means_partial_kernel(InitInputs in, int64_t N, double* partial)
{
    constexpr int M = NMEANS;
    __shared__ double sh[M][kMeansThreads / 32];
    double acc[M];
    for (int j = 0; j < M; ++j) acc[j] = 0.0;
    const int ia[6] = {0, 1, 2, 0, 0, 1}, ib[6] = {0, 1, 2, 1, 2, 2};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        double E[3], B[3];
        input_E(in, i, N, E);
        for (int a = 0; a < 3; ++a) B[a] = in.B[a * N + i];
        acc[0] += in.n[i];
        acc[1] += in.p[i];
        for (int a = 0; a < 3; ++a) {
            acc[2 + a] += E[a];
            acc[5 + a] += B[a];
        }
        for (int m = 0; m < 6; ++m) {
            acc[8 + m] += E[ia[m]] * E[ib[m]];
            acc[14 + m] += B[ia[m]] * B[ib[m]];
        }
        acc[20] += B[1] * E[2] - B[2] * E[1];
        acc[21] += B[2] * E[0] - B[0] * E[2];
        acc[22] += B[0] * E[1] - B[1] * E[0];
    }
    for (int j = 0; j < M; ++j)
        for (int o = 16; o > 0; o >>= 1) acc[j] += __shfl_down_sync(0xffffffffu, acc[j], o);
    if (threadIdx.x % 32 == 0)
        for (int j = 0; j < M; ++j) sh[j][threadIdx.x / 32] = acc[j];
    __syncthreads();
    if (threadIdx.x < M) {
        double a = 0.0;
        for (int w = 0; w < (int)(blockDim.x / 32); ++w) a += sh[threadIdx.x][w];
        partial[(int64_t)blockIdx.x * M + threadIdx.x] = a;
    }
}

__global__ void means_final_kernel(const double* partial, int nblocks, int64_t N, double* out)
{
    if (threadIdx.x < NMEANS) {
        double a = 0.0;
        for (int b = 0; b < nblocks; ++b) a += partial[(int64_t)b * NMEANS + threadIdx.x];
        out[threadIdx.x] = a / (double)N;
    }
}

// ---------------------------------------------------------------------------
// open boundaries: copy of the first interior cell (faces in order -x .. +z,
// which is the same as clamping every open-axis coordinate into [1, n-2])
// ---------------------------------------------------------------------------
// ---------------------------------------------------------------------------
// normal-B fix on one open face (axis a, side hi): B_n of the boundary cell is
// set so that the central-difference div B of the first interior cell
// vanishes; the change is carried by the h populations whose b is parallel to
// the normal (h_c += dB b_n / 8), and the f populations see the changed
// equilibrium through the collision (f_c += K_i [f_i^eq(new) - f_i^eq(old)]).
// ---------------------------------------------------------------------------
// f_c += K_i [f_i^eq(new) - f_i^eq(old)] for the 19 populations; `fv` holds
// their values, loaded before any store (the planes are distinct, which the
// compiler cannot prove); DIFF: qn holds the difference of the terms
template <int I, class Cfg, class R, bool DIFF = false>
struct FixF {
    static __device__ __forceinline__ void run(const PopView<Cfg>& V, int64_t c, const EqCell<R>& qo,
                                               const EqCell<R>& qn, const R* fv)
    {
        const R d = k_aw<I>(qo) * (DIFF ? feq_dev<I>(qn) : feq_dev<I>(qn) - feq_dev<I>(qo));
        st_pop<Cfg>(V.fg + fg_elem(I, 0, c, V.stride), fv[I] + d, V.hs.finv[I]);
        FixF<I + 1, Cfg, R, DIFF>::run(V, c, qo, qn, fv);
    }
};
template <class Cfg, class R, bool DIFF>
struct FixF<19, Cfg, R, DIFF> {
    static __device__ __forceinline__ void run(const PopView<Cfg>&, int64_t, const EqCell<R>&, const EqCell<R>&,
                                               const R*)
    {
    }
};

// nfaces = 1: the face `hi` of axis a; nfaces = 2: both faces of axis a in one
// launch (independent when the axis has at least 4 cells: a face writes its
// boundary layer and reads the two layers inside it)
// (the axis a is a template argument: with indices known at compile time nothing
// goes through local memory; float64, two cells: 18.5 -> 13.3 us)
template <class Cfg, int a>
__global__ void __launch_bounds__(128) bfix_kernel(PopView<Cfg> V, Phys<typename Cfg::real> k, int hi_first, int nfaces)
{
    grid_wait();  // (a programmatic launch: see the step kernel)
    using R = typename Cfg::real;
    const int n[3] = {V.nx, V.ny, V.nz};
    constexpr int a1 = (a + 1) % 3, a2 = (a + 2) % 3;
    const int64_t face = (int64_t)n[a1] * n[a2];
    const int64_t mm = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (mm >= nfaces * face) return;
    const int hi = nfaces == 2 ? (int)(mm / face) : hi_first;
    const int64_t m = mm % face;
    int q[3];
    q[a1] = (int)(m % n[a1]);
    q[a2] = (int)(m / n[a1]);
    const int sgn = hi ? -1 : 1;
    const int b = hi ? n[a] - 1 : 0;
    auto idx = [&](const int* r) { return r[0] + (int64_t)V.nx * (r[1] + (int64_t)V.ny * r[2]); };
    int r1[3] = {q[0], q[1], q[2]};
    r1[a] = b + sgn;
    R tang = R(0);
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const int ax = t == 0 ? a1 : a2;
        if (n[ax] == 1) continue;
        int rp[3] = {r1[0], r1[1], r1[2]}, rm[3] = {r1[0], r1[1], r1[2]};
        rp[ax] = wrap_coord(r1[ax] + 1, n[ax], V.periodic[ax]);
        rm[ax] = wrap_coord(r1[ax] - 1, n[ax], V.periodic[ax]);
        tang += ((R)V.prim[prim_elem(P_B + ax, idx(rp), V.stride)] - (R)V.prim[prim_elem(P_B + ax, idx(rm), V.stride)]) /
                (R(2) * k.dx);
    }
    int r2[3] = {q[0], q[1], q[2]};
    r2[a] = b + 2 * sgn;
    int rb[3] = {q[0], q[1], q[2]};
    rb[a] = b;
    const int64_t cb = idx(rb);
    const R Bfar = (R)V.prim[prim_elem(P_B + a, idx(r2), V.stride)];
    const R Bn_new = Bfar + R(sgn) * R(2) * k.dx * tang;
    Prim<R> so;
    load_prim<Cfg>(V.prim, V.stride, cb, so);
    R fv[19], hv[8];
#pragma unroll
    for (int i = 0; i < 19; ++i) fv[i] = ld_pop<Cfg>(V.fg + fg_elem(i, 0, cb, V.stride), V.hs.f[i]);
    constexpr int hp = plane_normal(0) == a ? 0 : (plane_normal(1) == a ? 1 : 2);  // the plane whose normal is axis a
#pragma unroll
    for (int j = 0; j < 8; ++j) hv[j] = (R)V.h[h_elem(8 * hp + j, cb, V.stride)];
    const R dB = Bn_new - so.B[a];
    Prim<R> sn = so;
    sn.B[a] = Bn_new;
    V.prim[prim_elem(P_B + a, cb, V.stride)] = (typename Cfg::prim)Bn_new;
    // h: populations of the plane whose normal is axis a, b = -/+ o_p n_hat
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const R bn = R(((j % 2) == 0 ? -1 : 1) * plane_orient(hp));
        V.h[h_elem(8 * hp + j, cb, V.stride)] = (typename Cfg::hpop)(hv[j] + dB * bn / R(8));
    }
    EqCell<R> qo, qn;
    if constexpr (sizeof(R) == 8) {
        // (the float64 rate again: one Lorentz factor for both, and the equilibria, linear
        // in the cell's terms, from the terms' differences)
        const R b2 = (so.u[0] * so.u[0] + so.u[1] * so.u[1] + so.u[2] * so.u[2]) * (k.inv_c * k.inv_c);
        Lorentz<R> lz;
        lz.g = rsqrt_newton(1.0 - b2);
        lz.g2 = lz.g * lz.g;
        lz.gm1 = lz.g2 * b2 * rcp_approx(lz.g + 1.0);
        R dE[3], dBo[3], dBn[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            dE[j] = so.E[j] - k.Er[j];
            dBo[j] = so.B[j] - k.Br[j];
            dBn[j] = sn.B[j] - k.Br[j];
        }
        eq_cell(so, so.n - k.n_r, so.eps - k.eps_r, dE, dBo, k, qo, &lz);
        eq_cell(sn, so.n - k.n_r, so.eps - k.eps_r, dE, dBn, k, qn, &lz);
        qn.f_rest -= qo.f_rest;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            qn.f_even_ax[j] -= qo.f_even_ax[j];
            qn.f_odd[j] -= qo.f_odd[j];
            qn.f_even_dg[j] -= qo.f_even_dg[j];
            qn.f_cross[j] -= qo.f_cross[j];
        }
        FixF<0, Cfg, R, true>::run(V, cb, qo, qn, fv);
    } else {
        eq_cell(so, k, qo);
        eq_cell(sn, k, qn);
        FixF<0, Cfg, R>::run(V, cb, qo, qn, fv);
    }
    grid_release();
}

// ---------------------------------------------------------------------------
// photospheric driving: the lowest `layers` z-layers are reset to the
// equilibrium of their own n, eps, B, rho_c with the two-vortex drive velocity
// (max |u| = u0) and E = -u x B
// ---------------------------------------------------------------------------
// the two-vortex drive velocity of column (x, y), (u_x, u_y) with max |u| = u0:
// tabulated once per run (it does not change in time)
__global__ void drive_profile_kernel(int nx, int ny, double u0, double* uv)
{
    const int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (m >= (int64_t)nx * ny) return;
    const int x = (int)(m % nx), y = (int)(m / nx);
    const double X = -3.0 + (x + 0.5) * 6.0 / nx;
    const double Y = -3.0 + (y + 0.5) * 6.0 / ny;
    const double xs = X < 0.0 ? X : X - 3.0;
    const double pi = 3.14159265358979323846;
    uv[2 * m] = u0 * sin(pi * xs / 3.0) * cos(pi * Y / 6.0);
    uv[2 * m + 1] = u0 * cos(pi * xs / 3.0) * sin(pi * Y / 6.0);
}

template <class Cfg>
__global__ void drive_kernel(PopView<Cfg> V, Phys<typename Cfg::real> k, int layers, const double* __restrict__ uv)
{
    using R = typename Cfg::real;
    const int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t plane = (int64_t)V.nx * V.ny;
    if (m >= plane * layers) return;
    const int64_t c = m, col = m % plane;
    Prim<R> s;
    load_prim<Cfg>(V.prim, V.stride, c, s);
    s.u[0] = (R)uv[2 * col];
    s.u[1] = (R)uv[2 * col + 1];
    s.u[2] = R(0);
    s.E[0] = -(s.u[1] * s.B[2] - s.u[2] * s.B[1]);
    s.E[1] = -(s.u[2] * s.B[0] - s.u[0] * s.B[2]);
    s.E[2] = -(s.u[0] * s.B[1] - s.u[1] * s.B[0]);
    store_prim<Cfg>(V.prim, V.stride, c, s);
    set_equilibrium<Cfg, R>(V, c, s, k);
}

// ---------------------------------------------------------------------------
// outputs
// ---------------------------------------------------------------------------
// component P of every cell's primitives into out (N values)
template <class Cfg>
__global__ void prim_component_kernel(PopView<Cfg> V, int P, typename Cfg::prim* out)
{
    const int64_t N = (int64_t)V.nx * V.ny * V.nz;
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c < N) out[c] = V.prim[prim_elem(P, c, V.stride)];
}


// Bound by the float64 rate, not by memory (176 bytes a cell in float32): ~35 float64
// instructions a cell, the conversions on the integer pipes. 1024^2 121 -> 65 us, 2048^2
// float16 475 -> 250 us.
template <class Cfg>
__global__ void __launch_bounds__(128) moments_kernel(PopView<Cfg> V, Phys<double> k, double* out)
{
    const int64_t N = (int64_t)V.nx * V.ny * V.nz;
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c >= N) return;
    Prim<double> s;
    {
        typename Cfg::real pv[NPRIM];
        ld_prims<Cfg>(V.prim + prim_elem(0, c, V.stride), V.stride, pv);
        s.n = widen(pv[P_N]);
        s.eps = widen(pv[P_EPS]);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            s.u[a] = widen(pv[P_U + a]);
            s.E[a] = widen(pv[P_E + a]);
            s.B[a] = widen(pv[P_B + a]);
        }
        s.rho = widen(pv[P_RHO]);
    }
    const double g = rsqrt_newton(1.0 - (s.u[0] * s.u[0] + s.u[1] * s.u[1] + s.u[2] * s.u[2]) * (k.inv_c * k.inv_c));
    double J[3];
    ohm_current_g(s.E, s.u, s.B, s.rho, g, k, J);
    out[0 * N + c] = s.n;
    out[1 * N + c] = k.gm1 * (s.eps - s.n * k.c2);
    out[2 * N + c] = s.eps;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        out[(3 + a) * N + c] = s.u[a];
        out[(6 + a) * N + c] = s.E[a];
        out[(9 + a) * N + c] = s.B[a];
        out[(13 + a) * N + c] = J[a];
    }
    out[12 * N + c] = s.rho;
}

// absolute post-collision populations (reference rest equilibrium added back)
template <class Cfg>
__global__ void populations_kernel(PopView<Cfg> V, RefPops ref, double* f, double* g, double* h)
{
    const int64_t N = (int64_t)V.nx * V.ny * V.nz;
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c >= N) return;
    for (int i = 0; i < 19; ++i) {
        if (f) f[i * N + c] = ref.f[i] + (double)ld_pop<Cfg>(V.fg + fg_elem(i, 0, c, V.stride), V.hs.f[i]);
        if (g) g[i * N + c] = ref.g[i] + (double)ld_pop<Cfg>(V.fg + fg_elem(i, 1, c, V.stride), V.hs.g[i]);
    }
    if (h)
        for (int i = 0; i < 25; ++i) h[i * N + c] = ref.h[i] + (double)V.h[h_elem(i, c, V.stride)];
}

// per-block float64 partial diagnostics: sum N^0, T^{0 nu} (4), rho_c, max |div B|,
// sum (div B)^2, non-finite count. A cell's sums over its populations and the
// sums over the 32 cells of a warp are taken in the storage's arithmetic type
// over the deviations (small numbers, rounded relative to themselves); the
// warp totals get the reference rest state of their cells and are summed
// over warps and blocks in float64. (float64 arithmetic per cell made this
// memory-bound pass bound by GB300's float64 rate, 15x slower.)
template <class Cfg>
__global__ void diag_kernel(PopView<Cfg> V, Phys<double> k, RefState r, double* partial)
{
    using R = typename Cfg::real;
    const int64_t N = (int64_t)V.nx * V.ny * V.nz;
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    R w[NPART] = {R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0)};  // deviations, |div B|, (div B)^2, bad
    if (c < N) {
        bool bad = false;
        R N0 = R(0), T0[4] = {R(0), R(0), R(0), R(0)}, rho = R(0);
        auto add = [&](int i, R fi, R gi) {
            bad = bad || !isfinite(fi) || !isfinite(gi);
            N0 += gi;
            T0[0] += fi;
#pragma unroll
            for (int a = 0; a < 3; ++a)
                if (c19(i, a)) T0[a + 1] += R(c19(i, a)) * fi;
        };
        {
            const V2<R> v = ld_fgpair<Cfg>(V.fg + fg_elem(0, 0, c, V.stride));
            add(0, Cfg::kHalf ? v.x * V.hs.f[0] : v.x, Cfg::kHalf ? v.y * V.hs.g[0] : v.y);
        }
#pragma unroll
        for (int i = 1; i < 19; i += 2) {
            const V4<R> v = ld_quad<Cfg>(V.fg + fg_elem(i, 0, c, V.stride));
            add(i, Cfg::kHalf ? v.x * V.hs.f[i] : v.x, Cfg::kHalf ? v.y * V.hs.g[i] : v.y);
            add(i + 1, Cfg::kHalf ? v.z * V.hs.f[i + 1] : v.z, Cfg::kHalf ? v.w * V.hs.g[i + 1] : v.w);
        }
#pragma unroll
        for (int m = 0; m < 12; ++m) {
            const V2<R> v = ld_hpair<Cfg>(V.h + h_elem(2 * m, c, V.stride));
            bad = bad || !isfinite(v.x) || !isfinite(v.y);
            rho += v.x;
            rho += v.y;
        }
        {
            const R hi = (R)V.h[h_elem(24, c, V.stride)];
            bad = bad || !isfinite(hi);
            rho += hi;
        }
        {
            R pv[NPRIM];
            ld_prims<Cfg>(V.prim + prim_elem(0, c, V.stride), V.stride, pv);
            for (int i = 0; i < NPRIM; ++i) bad = bad || !isfinite(pv[i]);
        }
        const int q[3] = {(int)(c % V.nx), (int)((c / V.nx) % V.ny), (int)(c / ((int64_t)V.nx * V.ny))};
        const int n[3] = {V.nx, V.ny, V.nz};
        R div = R(0);
        for (int a = 0; a < 3; ++a) {
            if (n[a] == 1) continue;
            int qp[3] = {q[0], q[1], q[2]}, qm[3] = {q[0], q[1], q[2]};
            qp[a] = wrap_coord(q[a] + 1, n[a], V.periodic[a]);
            qm[a] = wrap_coord(q[a] - 1, n[a], V.periodic[a]);
            const int64_t ip = qp[0] + (int64_t)V.nx * (qp[1] + (int64_t)V.ny * qp[2]);
            const int64_t im = qm[0] + (int64_t)V.nx * (qm[1] + (int64_t)V.ny * qm[2]);
            div += (R)V.prim[prim_elem(P_B + a, ip, V.stride)] - (R)V.prim[prim_elem(P_B + a, im, V.stride)];
        }
        div = div / (R(2) * (R)k.dx);
        w[0] = N0;
        for (int a = 0; a < 4; ++a) w[1 + a] = T0[a];
        w[5] = rho;
        w[6] = fabs(div);
        w[7] = div * div;
        w[8] = bad ? R(1) : R(0);
    }
    // the warp's cells in the arithmetic type (index 6 a max, the others sums)
#pragma unroll
    for (int j = 0; j < NPART; ++j)
        for (int o = 16; o > 0; o >>= 1) {
            const R other = __shfl_down_sync(0xffffffffu, w[j], o);
            w[j] = (j == 6) ? fmax(w[j], other) : w[j] + other;
        }
    __shared__ double sh[kDiagThreads / 32][NPART];
    const int wid = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (lane == 0) {
        const int64_t first = c;  // the warp's first cell
        const double cells = (double)(first >= N ? 0 : (N - first < 32 ? N - first : 32));
        for (int j = 0; j < NPART; ++j) sh[wid][j] = (double)w[j];
        sh[wid][0] += cells * r.n_r;  // reference rest state of the warp's cells
        sh[wid][1] += cells * r.eps_r;
        for (int a = 0; a < 3; ++a) sh[wid][2 + a] *= kQ;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int j = 0; j < NPART; ++j) {
            double acc = sh[0][j];
            for (int ww = 1; ww < (int)(blockDim.x / 32); ++ww) acc = (j == 6) ? fmax(acc, sh[ww][j]) : acc + sh[ww][j];
            partial[(int64_t)blockIdx.x * NPART + j] = acc;
        }
    }
}

__global__ void diag_final_kernel(const double* partial, int64_t nblocks, int64_t ncells, double* out)
{
    double v[NPART] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int64_t b = threadIdx.x; b < nblocks; b += blockDim.x) {
        for (int j = 0; j < NPART; ++j) {
            const double x = partial[b * NPART + j];
            v[j] = (j == 6) ? fmax(v[j], x) : v[j] + x;
        }
    }
    block_reduce_partials(v, out);
    __syncthreads();
    if (threadIdx.x == 0) {
        // out layout of the C ABI: sums, max |div B|, rms div B, non-finite count, cells
        const double sumsq = out[7];
        out[7] = sqrt(sumsq / (double)ncells);
        out[9] = (double)ncells;
    }
}

// ---------------------------------------------------------------------------
// reconnection rate at the null point (Sec. IV, KH-driven reconnection):
// argmin of B_x^2 + B_y^2 over rows [y_lo, y_hi) of a 2-D run, ties to the
// lowest cell index (the reduction is exact, so its order does not matter)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void min_pair(double& v, long long& i, double v2, long long i2)
{
    if (v2 < v || (v2 == v && i2 < i)) {
        v = v2;
        i = i2;
    }
}

__device__ __forceinline__ void block_min_pair(double& v, long long& i)
{
    __shared__ double sv[32];
    __shared__ long long si[32];
    for (int o = 16; o > 0; o >>= 1)
        min_pair(v, i, __shfl_down_sync(0xffffffffu, v, o), __shfl_down_sync(0xffffffffu, i, o));
    const int w = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (lane == 0) {
        sv[w] = v;
        si[w] = i;
    }
    __syncthreads();
    if (w == 0) {
        const int nw = (int)(blockDim.x / 32);
        v = lane < nw ? sv[lane] : CUDART_INF;
        i = lane < nw ? si[lane] : LLONG_MAX;
        for (int o = 16; o > 0; o >>= 1)
            min_pair(v, i, __shfl_down_sync(0xffffffffu, v, o), __shfl_down_sync(0xffffffffu, i, o));
    }
}

template <class Cfg>
__global__ void null_partial_kernel(PopView<Cfg> V, int y_lo, int y_hi, double* part_v, long long* part_i)
{
    const int64_t nb = (int64_t)V.nx * (y_hi - y_lo);
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    double v = CUDART_INF;
    long long i = LLONG_MAX;
    if (t < nb) {
        const long long c = (long long)y_lo * V.nx + t;
        const double bx = (double)V.prim[prim_elem(P_B, c, V.stride)], by = (double)V.prim[prim_elem(P_B + 1, c, V.stride)];
        const double b2 = __dadd_rn(__dmul_rn(bx, bx), __dmul_rn(by, by));  // no FMA: rounds as written
        if (b2 == b2) {  // NaN never wins
            v = b2;
            i = c;
        }
    }
    block_min_pair(v, i);
    if (threadIdx.x == 0) {
        part_v[blockIdx.x] = v;
        part_i[blockIdx.x] = i;
    }
}

// out: R, x, y, |B| at the null (NaN when the band holds no finite field)
template <class Cfg>
__global__ void null_final_kernel(const double* part_v, const long long* part_i, int64_t nblocks, PopView<Cfg> V,
                                  const typename Cfg::prim* ez0, double B0, double* out)
{
    double v = CUDART_INF;
    long long i = LLONG_MAX;
    for (int64_t b = threadIdx.x; b < nblocks; b += blockDim.x) min_pair(v, i, part_v[b], part_i[b]);
    block_min_pair(v, i);
    if (threadIdx.x == 0) {
        const int64_t N = (int64_t)V.nx * V.ny;
        if (i >= 0 && i < N) {
            const double ez = (double)V.prim[prim_elem(P_E + 2, i, V.stride)];
            out[0] = (ez - (double)ez0[i]) / B0;
            out[1] = (double)(i % V.nx);
            out[2] = (double)(i / V.nx);
            out[3] = sqrt(v);
        } else {
            out[0] = out[1] = out[2] = out[3] = CUDART_NAN;
        }
    }
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
static inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

template <class Cfg>
cudaError_t launch_init(const PopView<Cfg>& V, const InitInputs& in, const Phys<double>& k, int* bad,
                        cudaStream_t s)
{
    const int64_t N = (int64_t)V.nx * V.ny * V.nz;
    init_kernel<Cfg><<<blocks_for(N, 128), 128, 0, s>>>(V, in, init_phys(k, typename InitReal<Cfg>::type{}), init_consts(k),
                                                        bad);
    return cudaGetLastError();
}

cudaError_t launch_means(const InitInputs& in, int64_t N, double* partial, double* out, cudaStream_t s)
{
    int nb = (int)((N + kMeansThreads - 1) / kMeansThreads);
    nb = nb < kMeansBlocks ? nb : kMeansBlocks;
    means_partial_kernel<<<nb, kMeansThreads, 0, s>>>(in, N, partial);
    means_final_kernel<<<1, 32, 0, s>>>(partial, nb, N, out);
    return cudaGetLastError();
}

cudaError_t launch_drive_profile(int nx, int ny, double u0, double* uv, cudaStream_t s)
{
    drive_profile_kernel<<<blocks_for((int64_t)nx * ny, 256), 256, 0, s>>>(nx, ny, u0, uv);
    return cudaGetLastError();
}

template <class Cfg>
cudaError_t launch_boundaries(const PopView<Cfg>& V, const Phys<typename Cfg::real>& k, const int* bc, int layers,
                              const double* drive_uv, bool overlap, cudaStream_t s)
{
    const int n[3] = {V.nx, V.ny, V.nz};
    cudaError_t err = cudaSuccess;
    cudaLaunchConfig_t cfg{};
    cfg.blockDim = dim3(128);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = overlap ? 1 : 0;
    // (the copy of the interior neighbour into the open faces is done by the
    // step kernel itself; here the normal-B fix and the driving follow it)
    for (int a = 0; a < 3; ++a) {
        const bool lo = bc[2 * a] != 0 && n[a] >= 3, hi = bc[2 * a + 1] != 0 && n[a] >= 3;
        const int64_t m = (int64_t)n[(a + 1) % 3] * n[(a + 2) % 3];
        auto fix = [&](int64_t cells, int hi_first, int nfaces) {
            cfg.gridDim = dim3(blocks_for(cells, 128));
            const cudaError_t e = cudaLaunchKernelEx(
                &cfg, a == 0 ? bfix_kernel<Cfg, 0> : (a == 1 ? bfix_kernel<Cfg, 1> : bfix_kernel<Cfg, 2>), V, k, hi_first, nfaces);
            if (err == cudaSuccess) err = e;
        };
        if (lo && hi && n[a] >= 4) {
            fix(2 * m, 0, 2);
        } else {
            if (lo) fix(m, 0, 1);
            if (hi) fix(m, 1, 1);
        }
    }
    if (bc[4] == 2 && layers > 0 && drive_uv) {
        const int nl = layers < V.nz ? layers : V.nz;
        drive_kernel<Cfg><<<blocks_for((int64_t)V.nx * V.ny * nl, 128), 128, 0, s>>>(V, k, nl, drive_uv);
    }
    const cudaError_t last = cudaGetLastError();
    return err != cudaSuccess ? err : last;
}

template <class Cfg>
cudaError_t launch_moments(const PopView<Cfg>& V, const Phys<double>& k, double* out, cudaStream_t s)
{
    const int64_t N = (int64_t)V.nx * V.ny * V.nz;
    moments_kernel<Cfg><<<blocks_for(N, 128), 128, 0, s>>>(V, k, out);
    return cudaGetLastError();
}

template <class Cfg>
cudaError_t launch_prim_component(const PopView<Cfg>& V, int P, typename Cfg::prim* out, cudaStream_t s)
{
    const int64_t N = (int64_t)V.nx * V.ny * V.nz;
    prim_component_kernel<Cfg><<<blocks_for(N, 256), 256, 0, s>>>(V, P, out);
    return cudaGetLastError();
}

template <class Cfg>
cudaError_t launch_populations(const PopView<Cfg>& V, const RefPops& ref, double* f, double* g, double* h,
                               cudaStream_t s)
{
    const int64_t N = (int64_t)V.nx * V.ny * V.nz;
    populations_kernel<Cfg><<<blocks_for(N, 128), 128, 0, s>>>(V, ref, f, g, h);
    return cudaGetLastError();
}

template <class Cfg>
cudaError_t launch_diag(const PopView<Cfg>& V, const Phys<double>& k, const RefState& r, double* partial,
                        int64_t max_blocks, double* out, cudaStream_t s)
{
    const int64_t N = (int64_t)V.nx * V.ny * V.nz;
    const int64_t nb = blocks_for(N, kDiagThreads);
    if (nb > max_blocks) return cudaErrorInvalidValue;
    diag_kernel<Cfg><<<(unsigned)nb, kDiagThreads, 0, s>>>(V, k, r, partial);
    diag_final_kernel<<<1, kDiagThreads, 0, s>>>(partial, nb, N, out);
    return cudaGetLastError();
}

template <class Cfg>
cudaError_t launch_null(const PopView<Cfg>& V, int y_lo, int y_hi, const typename Cfg::prim* ez0, double B0,
                        double* scratch, int64_t scratch_doubles, double* out, cudaStream_t s)
{
    const int64_t nb = blocks_for((int64_t)V.nx * (y_hi - y_lo), kDiagThreads);
    if (2 * nb > scratch_doubles) return cudaErrorInvalidValue;
    double* pv = scratch;
    long long* pi = reinterpret_cast<long long*>(scratch + nb);
    null_partial_kernel<Cfg><<<(unsigned)nb, kDiagThreads, 0, s>>>(V, y_lo, y_hi, pv, pi);
    null_final_kernel<Cfg><<<1, kDiagThreads, 0, s>>>(pv, pi, nb, V, ez0, B0, out);
    return cudaGetLastError();
}

// max |u|^2 of a state into out[0] (float64 bits, atomicMax; out[0] zeroed
// before), out[1] (the running maximum of the next step) zeroed
template <class Cfg>
__global__ void umax_state_kernel(PopView<Cfg> V, double* out)
{
    const int64_t N = (int64_t)V.nx * V.ny * V.nz;
    double m = 0.0;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < N; c += (int64_t)gridDim.x * blockDim.x) {
        double u2 = 0.0;
        for (int a = 0; a < 3; ++a) {
            const double u = (double)V.prim[prim_elem(P_U + a, c, V.stride)];
            u2 += u * u;
        }
        m = fmax(m, u2);
    }
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (threadIdx.x % 32 == 0) atomicMax(reinterpret_cast<unsigned long long*>(out), (unsigned long long)__double_as_longlong(m));
    if (blockIdx.x == 0 && threadIdx.x == 0) out[1] = 0.0;
}

// after a step: the running maximum becomes the input state's, and restarts
__global__ void umax_roll_kernel(double* u)
{
    u[0] = u[1];
    u[1] = 0.0;
}

// E of a state into both history planes E_{k-1}, E_{k-2} (3 N float64 each)
template <class Cfg>
__global__ void relax_history_kernel(PopView<Cfg> V, double* e)
{
    const int64_t N = (int64_t)V.nx * V.ny * V.nz;
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c >= N) return;
    for (int a = 0; a < 3; ++a) {
        const double E = (double)V.prim[prim_elem(P_E + a, c, V.stride)];
        e[a * N + c] = E;
        e[(3 + a) * N + c] = E;
    }
}

template <class Cfg>
cudaError_t launch_umax_state(const PopView<Cfg>& V, double* out, cudaStream_t s)
{
    const int64_t N = (int64_t)V.nx * V.ny * V.nz;
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(double), s);
    if (e != cudaSuccess) return e;
    const int64_t nb = blocks_for(N, 256);
    umax_state_kernel<Cfg><<<(unsigned)(nb < 1216 ? nb : 1216), 256, 0, s>>>(V, out);
    return cudaGetLastError();
}

cudaError_t launch_umax_roll(double* u, cudaStream_t s)
{
    umax_roll_kernel<<<1, 1, 0, s>>>(u);
    return cudaGetLastError();
}

template <class Cfg>
cudaError_t launch_relax_history(const PopView<Cfg>& V, double* e, cudaStream_t s)
{
    const int64_t N = (int64_t)V.nx * V.ny * V.nz;
    relax_history_kernel<Cfg><<<blocks_for(N, 256), 256, 0, s>>>(V, e);
    return cudaGetLastError();
}

#define LB_INSTANTIATE(CFG)                                                                                        \
    template cudaError_t launch_init<CFG>(const PopView<CFG>&, const InitInputs&, const Phys<double>&, int*,      \
                                          cudaStream_t);                                                           \
    template cudaError_t launch_boundaries<CFG>(const PopView<CFG>&, const Phys<CFG::real>&, const int*, int,      \
                                                const double*, bool, cudaStream_t);                                      \
    template cudaError_t launch_moments<CFG>(const PopView<CFG>&, const Phys<double>&, double*, cudaStream_t);     \
    template cudaError_t launch_prim_component<CFG>(const PopView<CFG>&, int, CFG::prim*, cudaStream_t);           \
    template cudaError_t launch_populations<CFG>(const PopView<CFG>&, const RefPops&, double*, double*, double*,  \
                                                 cudaStream_t);                                                    \
    template cudaError_t launch_diag<CFG>(const PopView<CFG>&, const Phys<double>&, const RefState&, double*,      \
                                          int64_t, double*, cudaStream_t);                                         \
    template cudaError_t launch_null<CFG>(const PopView<CFG>&, int, int, const CFG::prim*, double, double*,       \
                                          int64_t, double*, cudaStream_t);                                         \
    template cudaError_t launch_umax_state<CFG>(const PopView<CFG>&, double*, cudaStream_t);                      \
    template cudaError_t launch_relax_history<CFG>(const PopView<CFG>&, double*, cudaStream_t);

LB_INSTANTIATE(CfgF64)
LB_INSTANTIATE(CfgF32)
LB_INSTANTIATE(CfgF16)

}  // namespace lb
