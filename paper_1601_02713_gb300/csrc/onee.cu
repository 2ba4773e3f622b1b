// One-electron integrals (overlap, kinetic, nuclear attraction), their
// derivatives for the analytic gradient, primitive-pair data, the nuclear
// repulsion, and the Boys table.
//
// Obara-Saika recursions (Obara & Saika, J. Chem. Phys. 84, 3963 (1986)),
// one direction at a time for the overlap,
//   S(i+1, j) = PA S(i, j) + [i S(i-1, j) + j S(i, j-1)] / (2p),
//   S(i, j+1) = PB S(i, j) + [i S(i-1, j) + j S(i, j-1)] / (2p),
// the kinetic energy as (1/2) <grad a | grad b>,
//   T(i, j) = 1/2 [ i j S(i-1,j-1) - 2a j S(i+1,j-1) - 2b i S(i-1,j+1) + 4ab S(i+1,j+1) ],
// and the nuclear attraction with auxiliary orders m,
//   V^m(a+1_i, b) = PA_i V^m(a,b) - PC_i V^{m+1}(a,b)
//                   + a_i/(2p) [V^m(a-1_i,b) - V^{m+1}(a-1_i,b)] + b_i/(2p) [V^m(a,b-1_i) - V^{m+1}(a,b-1_i)],
//   V^m(0,0) = (2 pi / p) K F_m(p |PC|^2)     (and the same rule for b+1_i with PB).
#include <math.h>

#include <algorithm>

#include "eri_kernels.cuh"
#include "internal.h"
#include "nuclear.cuh"

namespace pimd {

namespace {

constexpr double kPi = 3.14159265358979323846;
__device__ __forceinline__ int cidx_host_dev(const int* e)
{
    const int l = e[0] + e[1] + e[2];
    return (l - e[0]) * (l - e[0] + 1) / 2 + e[2];
}

__device__ __forceinline__ void cart_of_d(int l, int idx, int* e)
{
    int n = 0;
    for (int x = l; x >= 0; x--)
        for (int y = l - x; y >= 0; y--) {
            if (n == idx) {
                e[0] = x;
                e[1] = y;
                e[2] = l - x - y;
                return;
            }
            n++;
        }
}

// 1-D overlap table S[i][j], i <= imax, j <= jmax (without the (pi/p)^{1/2} K factor)
__device__ void os_overlap_1d(int imax, int jmax, double PA, double PB, double p, double S[6][5])
{
    const double o2p = 0.5 / p;
    S[0][0] = 1.0;
    for (int i = 0; i <= imax; i++)
        for (int j = 0; j <= jmax; j++) {
            if (i == 0 && j == 0) continue;
            double v;
            if (i > 0) {
                v = PA * S[i - 1][j];
                if (i > 1) v += (i - 1) * o2p * S[i - 2][j];
                if (j > 0) v += j * o2p * S[i - 1][j - 1];
            } else {
                v = PB * S[i][j - 1];
                if (j > 1) v += (j - 1) * o2p * S[i][j - 2];
            }
            S[i][j] = v;
        }
}

__device__ __forceinline__ double kin_1d(const double S[6][5], int i, int j, double a, double b)
{
    double t = 4.0 * a * b * S[i + 1][j + 1];
    if (i > 0 && j > 0) t += i * j * S[i - 1][j - 1];
    if (j > 0) t -= 2.0 * a * j * S[i + 1][j - 1];
    if (i > 0) t -= 2.0 * b * i * S[i - 1][j + 1];
    return 0.5 * t;
}

// run(LA, LB) as compile-time constants for shells of angular momenta la, lb
template <class F>
__device__ __forceinline__ void by_l(int la, int lb, F&& run)
{
    using std::integral_constant;
    switch (3 * la + lb) {
    case 0: run(integral_constant<int, 0>(), integral_constant<int, 0>()); break;
    case 1: run(integral_constant<int, 0>(), integral_constant<int, 1>()); break;
    case 2: run(integral_constant<int, 0>(), integral_constant<int, 2>()); break;
    case 3: run(integral_constant<int, 1>(), integral_constant<int, 0>()); break;
    case 4: run(integral_constant<int, 1>(), integral_constant<int, 1>()); break;
    case 5: run(integral_constant<int, 1>(), integral_constant<int, 2>()); break;
    case 6: run(integral_constant<int, 2>(), integral_constant<int, 0>()); break;
    case 7: run(integral_constant<int, 2>(), integral_constant<int, 1>()); break;
    case 8: run(integral_constant<int, 2>(), integral_constant<int, 2>()); break;
    }
}

__global__ void pair_data_kernel(Pairs P, int* npp, double* pp, Shells S, BasisPrimDev B)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= P.n) return;
    const int a = P.sa[g], b = P.sb[g];
    const int pa = B.sprim[a], pb = B.sprim[b], na = B.snprim[a], nb = B.snprim[b];
    double AB2 = 0.0;
    double A[3], Bc[3];
    for (int x = 0; x < 3; x++) {
        A[x] = S.xyz[3 * a + x];
        Bc[x] = S.xyz[3 * b + x];
        AB2 += (A[x] - Bc[x]) * (A[x] - Bc[x]);
    }
    const double c0 = 1.4142135623730950488 * pow(kPi, 1.25);
    // primitive pairs whose prefactor is below 1e-17 of the pair's largest
    // one are dropped (their share of any integral is below double rounding)
    double kmax = 0.0;
    for (int i = 0; i < na; i++)
        for (int j = 0; j < nb; j++) {
            const double ea = B.exps[pa + i], eb = B.exps[pb + j];
            kmax = fmax(kmax, fabs(B.coefs[pa + i] * B.coefs[pb + j] * exp(-ea * eb / (ea + eb) * AB2) / (ea + eb)));
        }
    int k = 0;
    for (int i = 0; i < na; i++)
        for (int j = 0; j < nb; j++) {
            const double ea = B.exps[pa + i], eb = B.exps[pb + j];
            const double p = ea + eb, ip = 1.0 / p;
            const double kij = B.coefs[pa + i] * B.coefs[pb + j] * exp(-ea * eb * ip * AB2) * ip;
            if (fabs(kij) < 1e-17 * kmax) continue;
            const double Px = (ea * A[0] + eb * Bc[0]) * ip, Py = (ea * A[1] + eb * Bc[1]) * ip,
                         Pz = (ea * A[2] + eb * Bc[2]) * ip;
            const double vals[PP_NF] = {p,  Px, Py, Pz, c0 * kij, Px - A[0], Py - A[1], Pz - A[2],
                                        0.5 * ip, 0.5 * ip * ip, ea, eb};
            for (int f = 0; f < PP_NF; f++) pp[((size_t)f * PIMD_MAXPP + k) * P.n + g] = vals[f];
            k++;
        }
    npp[g] = k;
}

__device__ __forceinline__ double lane_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// primitive pair (i, j) of shells (sa, sb): exponents and Gaussian product
struct PrimPair {
    double a, b, p, K, P[3], PA[3], PB[3];
    __device__ __forceinline__ PrimPair(const Shells& S, const BasisPrimDev& B, int sa, int sb, int i, int j)
    {
        const int pa = B.sprim[sa] + i, pb = B.sprim[sb] + j;
        a = B.exps[pa];
        b = B.exps[pb];
        p = a + b;
        double AB2 = 0.0;
#pragma unroll
        for (int x = 0; x < 3; x++) {
            const double A = S.xyz[3 * sa + x], Bc = S.xyz[3 * sb + x];
            AB2 += (A - Bc) * (A - Bc);
            P[x] = (a * A + b * Bc) / p;
            PA[x] = P[x] - A;
            PB[x] = P[x] - Bc;
        }
        K = B.coefs[pa] * B.coefs[pb] * exp(-a * b / p * AB2);
    }
};

// F[m] = -Z_c (2 pi / p) K F_m(p |P - C|^2) of nucleus c, m = 0..L; PC = P - C
template <int L>
__device__ __forceinline__ void nuclear_boys(const PrimPair& g, const AtomsDev& At, int c, const double* boys,
                                             double PC[3], double* F)
{
    double r2 = 0.0;
#pragma unroll
    for (int x = 0; x < 3; x++) {
        PC[x] = g.P[x] - At.xyz[3 * c + x];
        r2 += PC[x] * PC[x];
    }
    boys_eval<L>(g.p * r2, boys, -At.Z[c] * 2.0 * kPi / g.p * g.K, F);
}

// S, T, V of one shell pair by one warp. The nuclear attraction is the work:
// (primitive pair, nucleus) is one lane's unit, 9 x 24 of them for (H2O)8, and
// its recursion straight-line code; the lanes' Cartesian blocks are summed over
// the warp. Bound by the latency of a lane's FP64 chain: one thread per pair
// with the recursion's tables in local memory, as before, took 12.8 ms for one
// bead of (H2O)8.
template <int LA, int LB>
__device__ __forceinline__ void one_e_pair(int g, const Pairs& P, const Shells& S, const BasisPrimDev& B,
                                           const AtomsDev& At, const Reps& R, double* Sm, double* Tm, double* Vm,
                                           const double* boys)
{
    constexpr int nac = ncart(LA), nbc = ncart(LB), n = nac * nbc;
    const int sa = P.sa[g], sb = P.sb[g], r = S.rep[sa], lane = threadIdx.x & 31;
    const int na = B.snprim[sa], np = na * B.snprim[sb];
    const int c0 = At.rep_atom0[r], nc = At.rep_atom0[r + 1] - c0;
    double Sb[n], Tb[n], Vb[n];
#pragma unroll
    for (int k = 0; k < n; k++) Sb[k] = Tb[k] = Vb[k] = 0.0;
    for (int u = lane; u < np * nc; u += 32) {
        const PrimPair q(S, B, sa, sb, (u % np) % na, (u % np) / na);
        double PC[3], F[LA + LB + 1];
        nuclear_boys<LA + LB>(q, At, c0 + u / np, boys, PC, F);
        nuc_of<LA, LB>(F, q.PA, q.PB, PC, 0.5 / q.p, Vb);
    }
    if (lane < np) {
        const PrimPair q(S, B, sa, sb, lane % na, lane / na);
        double S1[3][6][5];
        for (int x = 0; x < 3; x++) os_overlap_1d(LA + 1, LB + 1, q.PA[x], q.PB[x], q.p, S1[x]);
        const double pre = q.K * pow(kPi / q.p, 1.5);
        for (int ia = 0; ia < nac; ia++) {
            int e[3];
            cart_of_d(LA, ia, e);
            for (int ib = 0; ib < nbc; ib++) {
                int f[3];
                cart_of_d(LB, ib, f);
                const double sx = S1[0][e[0]][f[0]], sy = S1[1][e[1]][f[1]], sz = S1[2][e[2]][f[2]];
                const double tx = kin_1d(S1[0], e[0], f[0], q.a, q.b), ty = kin_1d(S1[1], e[1], f[1], q.a, q.b),
                             tz = kin_1d(S1[2], e[2], f[2], q.a, q.b);
                Sb[ia * nbc + ib] = pre * sx * sy * sz;
                Tb[ia * nbc + ib] = pre * (tx * sy * sz + sx * ty * sz + sx * sy * tz);
            }
        }
    }
    const int N = R.nbf[r];
    const size_t off = R.moff[r];
    const int fa = S.bf[sa], fb = S.bf[sb];
    double* const out[3] = {Sm, Tm, Vm};
    double* const in[3] = {Sb, Tb, Vb};
#pragma unroll
    for (int k = 0; k < 3; k++) {
        double c[n], t[n];
#pragma unroll
        for (int e = 0; e < n; e++) c[e] = lane_sum(in[k][e]);
        sph_index<1, LA, nbc>(c, t);
        sph_index<nsph(LA), LB, 1>(t, c);
        if (lane == 0)
#pragma unroll
            for (int i = 0; i < nsph(LA); i++)
#pragma unroll
                for (int j = 0; j < nsph(LB); j++) {
                    out[k][off + (size_t)(fa + i) * N + fb + j] = c[i * nsph(LB) + j];
                    out[k][off + (size_t)(fb + j) * N + fa + i] = c[i * nsph(LB) + j];
                }
    }
}

// one warp per pair
__global__ void __launch_bounds__(64) one_e_kernel(Pairs P, Shells S, BasisPrimDev B, AtomsDev At, Reps R, double* Sm,
                                                   double* Tm, double* Vm, const double* boys)
{
    const int g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (g >= P.n) return;
    const int la = S.l[P.sa[g]], lb = S.l[P.sb[g]];
    auto run = [&](auto a, auto b) {
        one_e_pair<decltype(a)::value, decltype(b)::value>(g, P, S, B, At, R, Sm, Tm, Vm, boys);
    };
    by_l(la, lb, run);
}

// derivative of the bra Gaussian: d/dA_x g_a = 2 alpha g_{a+1_x} - a_x g_{a-1_x},
// of one (pair, orientation) by one warp. Every term is contracted with the
// density as soon as it is made, so a lane keeps three sums instead of
// derivative blocks. Nuclear attraction: the lanes take the nuclei, G lanes to
// a nucleus (its primitive pairs split over them) where there are fewer than
// 32; one bead of (H2O)8 with a thread per (pair, orientation): 62.7 ms.
template <int LA, int LB>
__device__ __forceinline__ void grad_1e_pair(int sa, int sb, const Shells& S, const BasisPrimDev& B,
                                             const AtomsDev& At, const Reps& R, const double* D, const double* W,
                                             double* grad, const double* boys, double fxs)
{
    constexpr int nac = ncart(LA), nbc = ncart(LB), nas = nsph(LA), nbs = nsph(LB);
    const int r = S.rep[sa], N = R.nbf[r], lane = threadIdx.x & 31;
    const size_t off = R.moff[r] + (size_t)S.bf[sa] * N + S.bf[sb];
    const int na = B.snprim[sa], np = na * B.snprim[sb];
    // density block in Cartesian-component form (sum_sph X_s I_s = sum_cart X_c I_c)
    auto load = [&](const double* M, double* c) {
        double t[nac * nbc];
#pragma unroll
        for (int i = 0; i < nas; i++)
#pragma unroll
            for (int j = 0; j < nbs; j++) c[i * nbs + j] = __ldg(M + off + (size_t)i * N + j);
        sph_index_t<1, LA, nbs>(c, t);
        sph_index_t<nac, LB, 1>(t, c);
    };
    double Dc[nac * nbc];
    load(D, Dc);
    double ga[3] = {0.0, 0.0, 0.0};
    // nuclear attraction: basis-function term on the bra atom and, by
    // translational invariance of the three-centre integral (dA + dB + dC = 0,
    // the ket term equal to the bra term by symmetry), the operator term
    // -2 sum D dV^C/dA on nucleus C itself
    const int c0 = At.rep_atom0[r], nc = At.rep_atom0[r + 1] - c0;
    const int G = nc >= 32 ? 1 : nc >= 16 ? 2 : nc >= 8 ? 4 : nc >= 4 ? 8 : 16;
    for (int cb = 0; cb < nc; cb += 32 / G) {
        const int c = cb + lane / G;
        double s[3] = {0.0, 0.0, 0.0};
        if (c < nc)
            for (int k = lane % G; k < np; k += G) {
                const PrimPair q(S, B, sa, sb, k % na, k / na);
                double PC[3], F[LA + LB + 2];
                nuclear_boys<LA + LB + 1>(q, At, c0 + c, boys, PC, F);
                nuc_grad_of<LA, LB>(F, q.PA, q.PB, PC, 0.5 / q.p, 2.0 * q.a, Dc, s);
            }
#pragma unroll
        for (int x = 0; x < 3; x++) {
            s[x] *= 2.0;
            for (int o = 1; o < G; o <<= 1) s[x] += __shfl_xor_sync(0xffffffffu, s[x], o);
            if (c < nc && lane % G == 0) {
                ga[x] += s[x];
                det_add(grad + 3 * (c0 + c) + x, -s[x], fxs);
            }
        }
    }
    // overlap and kinetic energy: a lane per primitive pair
    if (lane < np) {
        double Wc[nac * nbc];
        load(W, Wc);
        const PrimPair q(S, B, sa, sb, lane % na, lane / na);
        double S1[3][6][5];
        for (int x = 0; x < 3; x++) os_overlap_1d(LA + 2, LB + 1, q.PA[x], q.PB[x], q.p, S1[x]);
        const double pre = 2.0 * q.K * pow(kPi / q.p, 1.5);
        // components of level LA + 1 with weight 2 alpha, of level LA - 1 with -a_x
        for (int lev = 0; lev < (LA > 0 ? 2 : 1); lev++) {
            const int lq = lev == 0 ? LA + 1 : LA - 1;
            for (int iq = 0; iq < ncart(lq); iq++) {
                int e[3];
                cart_of_d(lq, iq, e);
                for (int ib = 0; ib < nbc; ib++) {
                    int f[3];
                    cart_of_d(LB, ib, f);
                    const double sx = S1[0][e[0]][f[0]], sy = S1[1][e[1]][f[1]], sz = S1[2][e[2]][f[2]];
                    const double tx = kin_1d(S1[0], e[0], f[0], q.a, q.b), ty = kin_1d(S1[1], e[1], f[1], q.a, q.b),
                                 tz = kin_1d(S1[2], e[2], f[2], q.a, q.b);
                    const double sv = pre * sx * sy * sz;
                    const double tv = pre * (tx * sy * sz + sx * ty * sz + sx * sy * tz);
#pragma unroll
                    for (int x = 0; x < 3; x++) {
                        // the component this one is the x-derivative of
                        int d[3] = {e[0], e[1], e[2]};
                        d[x] += lev == 0 ? -1 : 1;
                        if (d[x] < 0) continue;
                        const int k = cidx_host_dev(d) * nbc + ib;
                        ga[x] += (lev == 0 ? 2.0 * q.a : -(double)d[x]) * (Dc[k] * tv - Wc[k] * sv);
                    }
                }
            }
        }
    }
    const int atom_a = S.atom[sa];
#pragma unroll
    for (int x = 0; x < 3; x++) {
        const double v = lane_sum(ga[x]);
        if (lane == 0) det_add(grad + 3 * atom_a + x, v, fxs);
    }
}

// one warp per (pair, orientation)
__global__ void __launch_bounds__(64) grad_1e_kernel(Pairs P, Shells S, BasisPrimDev B, AtomsDev At, Reps R,
                                                     const double* D, const double* W, double* grad,
                                                     const double* boys, double fxs)
{
    const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t >= 2 * P.n) return;
    int sa = P.sa[t >> 1], sb = P.sb[t >> 1];
    if (t & 1) {
        if (sa == sb) return;
        const int tmp = sa;
        sa = sb;
        sb = tmp;
    }
    auto run = [&](auto a, auto b) {
        grad_1e_pair<decltype(a)::value, decltype(b)::value>(sa, sb, S, B, At, R, D, W, grad, boys, fxs);
    };
    by_l(S.l[sa], S.l[sb], run);
}

__global__ void vnn_kernel(AtomsDev At, int natom, const int* atom_rep, double* enn, double* grad, double fxs)
{
    const int A = blockIdx.x * blockDim.x + threadIdx.x;
    if (A >= natom) return;
    const int r = atom_rep[A];
    const int c0 = At.rep_atom0[r], c1 = At.rep_atom0[r + 1];
    double e = 0.0, g[3] = {0.0, 0.0, 0.0};
    for (int Bi = c0; Bi < c1; Bi++) {
        if (Bi == A) continue;
        double d[3], r2 = 0.0;
        for (int x = 0; x < 3; x++) {
            d[x] = At.xyz[3 * A + x] - At.xyz[3 * Bi + x];
            r2 += d[x] * d[x];
        }
        const double rr = sqrt(r2);
        const double zz = At.Z[A] * At.Z[Bi];
        e += 0.5 * zz / rr;
        for (int x = 0; x < 3; x++) g[x] -= zz * d[x] / (rr * r2);
    }
    det_add(enn + r, e, fxs);
    if (grad)
        for (int x = 0; x < 3; x++) det_add(grad + 3 * A + x, g[x], fxs);
}

__global__ void boys_eval_kernel(int n, int m, const double* T, double* F, const double* boys)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double t = T[i];
    // the table covers T >= 0 only: a negative or non-finite argument gives NaN
    if (!(t >= 0.0) || !isfinite(t)) {
        F[i] = nan("");
        return;
    }
    double f[BOYS_MMAX + 1];
    boys_eval_n(m, t, boys, 1.0, f);
    F[i] = f[m];
}

// FP32 evaluation of the mixed-precision quartets: variant 0 the
// compile-time-order form of the straight-line kernels, 1 the runtime-order
// form of the cooperative kernels
template <int L>
__device__ __forceinline__ float boys_f32_fixed(float t, const float* boysf)
{
    float f[L + 1];
    boys_eval<L>(t, boysf, 1.0f, f);
    return f[L];
}

__global__ void boys_eval_f32_kernel(int n, int m, const float* T, float* F, const float* boysf, int variant)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float t = T[i];
    if (!(t >= 0.0f) || !isfinite(t)) {
        F[i] = nanf("");
        return;
    }
    if (variant == 1) {
        float f[BOYS_MMAX + 1];
        boys_eval_n(m, t, boysf, 1.0f, f);
        F[i] = f[m];
        return;
    }
    float v = 0.0f;
    switch (m) {
    case 0: v = boys_f32_fixed<0>(t, boysf); break;
    case 1: v = boys_f32_fixed<1>(t, boysf); break;
    case 2: v = boys_f32_fixed<2>(t, boysf); break;
    case 3: v = boys_f32_fixed<3>(t, boysf); break;
    case 4: v = boys_f32_fixed<4>(t, boysf); break;
    case 5: v = boys_f32_fixed<5>(t, boysf); break;
    case 6: v = boys_f32_fixed<6>(t, boysf); break;
    case 7: v = boys_f32_fixed<7>(t, boysf); break;
    case 8: v = boys_f32_fixed<8>(t, boysf); break;
    case 9: v = boys_f32_fixed<9>(t, boysf); break;
    case 10: v = boys_f32_fixed<10>(t, boysf); break;
    case 11: v = boys_f32_fixed<11>(t, boysf); break;
    default: v = boys_f32_fixed<12>(t, boysf); break;
    }
    F[i] = v;
}

}  // namespace

void launch_boys_eval_f32(int n, int m, const float* T, float* F, const float* boysf, int variant, cudaStream_t st)
{
    if (n == 0) return;
    boys_eval_f32_kernel<<<(n + 127) / 128, 128, 0, st>>>(n, m, T, F, boysf, variant);
}

void launch_pair_data(const Pairs& P, int* npp, double* pp, const Shells& S, const BasisPrimDev& B,
                      cudaStream_t st)
{
    if (P.n == 0) return;
    pair_data_kernel<<<(P.n + 127) / 128, 128, 0, st>>>(P, npp, pp, S, B);
}

void launch_one_electron(const Pairs& P, const Shells& S, const BasisPrimDev& B, const AtomsDev& At,
                         const Reps& R, double* Sm, double* Tm, double* Vm, const double* boys, cudaStream_t st)
{
    if (P.n == 0) return;
    one_e_kernel<<<(P.n + 1) / 2, 64, 0, st>>>(P, S, B, At, R, Sm, Tm, Vm, boys);
}

void launch_grad_1e(const Pairs& P, const Shells& S, const BasisPrimDev& B, const AtomsDev& At, const Reps& R,
                    const double* D, const double* W, double* grad, const double* boys, double fxs,
                    cudaStream_t st)
{
    if (P.n == 0) return;
    grad_1e_kernel<<<P.n, 64, 0, st>>>(P, S, B, At, R, D, W, grad, boys, fxs);
}

void launch_vnn(const AtomsDev& At, int natom_total, const int* atom_rep, double* enn, double* grad,
                cudaStream_t st, double fxs)
{
    if (natom_total == 0) return;
    vnn_kernel<<<(natom_total + 127) / 128, 128, 0, st>>>(At, natom_total, atom_rep, enn, grad, fxs);
}

void launch_boys_eval(int n, int m, const double* T, double* F, const double* boys, cudaStream_t st)
{
    if (n == 0) return;
    boys_eval_kernel<<<(n + 127) / 128, 128, 0, st>>>(n, m, T, F, boys);
}

// F_m(T) = e^{-T} sum_i (2T)^i / ((2m+1)(2m+3)...(2m+2i+1)), a sum of positive
// terms evaluated in long double; stored as F_{m+j}(T_k) / j! and e^{-T_k}.
void boys_fill_table(double* tab)
{
    const int NM = BOYS_MT + BOYS_NTAYLOR;
    long double F[BOYS_MT + BOYS_NTAYLOR];
    for (int k = 0; k < BOYS_NT; k++) {
        const long double T = (long double)k / BOYS_GRID;
        for (int m = 0; m < NM; m++) {
            long double term = 1.0L / (2 * m + 1), sum = term;
            for (int i = 1; i < 2000; i++) {
                term *= 2.0L * T / (2 * m + 2 * i + 1);
                sum += term;
                if (term < 1e-22L * sum) break;
            }
            F[m] = expl(-T) * sum;
        }
        long double fact = 1.0L;
        for (int j = 0; j < BOYS_NTAYLOR; j++) {
            if (j > 0) fact *= j;
            for (int m = 0; m < BOYS_MT; m++)
                tab[((size_t)k * BOYS_MT + m) * BOYS_NTAYLOR + j] = (double)(F[m + j] / fact);
        }
    }
    for (int k = 0; k < BOYS_NE; k++) tab[BOYS_EXP_OFF + k] = (double)expl(-(long double)k / BOYS_GRID);
}

void boys_table_upload(double** dev_tab, float** dev_tabf, dfloat** dev_tabd)
{
    static double host[BOYS_TAB_DOUBLES];
    static float hostf[BOYS_TAB_FLOATS];
    static bool filled = false;
    if (!filled) {
        boys_fill_table(host);
        for (int k = 0; k < BOYS_NT; k++) {
            for (int m = 0; m < BOYS_MT; m++)
                for (int j = 0; j < BOYS_NTAYLOR_F; j++)
                    hostf[((size_t)k * BOYS_MT + m) * BOYS_NTAYLOR_F + j] =
                        (float)host[((size_t)k * BOYS_MT + m) * BOYS_NTAYLOR + j];
            hostf[(size_t)BOYS_NT * BOYS_MT * BOYS_NTAYLOR_F + k] = (float)host[(size_t)BOYS_NT * BOYS_MT * BOYS_NTAYLOR + k];
        }
        filled = true;
    }
    cudaMalloc(dev_tab, sizeof(host));
    cudaMemcpy(*dev_tab, host, sizeof(host), cudaMemcpyHostToDevice);
    cudaMalloc(dev_tabf, sizeof(hostf));
    cudaMemcpy(*dev_tabf, hostf, sizeof(hostf), cudaMemcpyHostToDevice);
    cudaMalloc(dev_tabd, sizeof(dfloat) * BOYS_TAB_DOUBLES);
    launch_to_dfloat(*dev_tab, *dev_tabd, BOYS_TAB_DOUBLES, nullptr);
    cudaStreamSynchronize(nullptr);
}

__global__ void to_dfloat_kernel(const double* src, dfloat* dst, long long n)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = dfloat(src[i]);
}

void launch_to_dfloat(const double* src, dfloat* dst, long long n, cudaStream_t st)
{
    if (n <= 0) return;
    to_dfloat_kernel<<<(int)std::min<long long>((n + 255) / 256, 1024), 256, 0, st>>>(src, dst, n);
}

__global__ void any_above_kernel(const double* v, long long n, double lim, int* flag)
{
    bool any = false;
    for (long long i = threadIdx.x; i < n; i += blockDim.x) any = any || !(fabs(v[i]) <= lim);
    const int f = __syncthreads_or(any);
    if (threadIdx.x == 0) *flag = f != 0;
}

void launch_any_above(const double* v, long long n, double lim, int* flag, cudaStream_t st)
{
    any_above_kernel<<<1, 256, 0, st>>>(v, n, lim, flag);
}

__global__ void pair_dfloat_kernel(Pairs P, Shells S, dfloat* ppd, dfloat* abd)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= P.n) return;
    const size_t n = P.n;
    const int sa = P.sa[g], sb = P.sb[g], np = P.npp[g];
    for (int x = 0; x < 3; x++) abd[x * n + g] = dfloat(S.xyz[3 * sa + x] - S.xyz[3 * sb + x]);
    for (int k = 0; k < np; k++) {
        for (int f = 0; f < PP_NF; f++)
            ppd[((size_t)f * PIMD_MAXPP + k) * n + g] = dfloat(P.pp[((size_t)f * PIMD_MAXPP + k) * n + g]);
        for (int x = 0; x < 3; x++)
            ppd[((size_t)(PP_PBX + x) * PIMD_MAXPP + k) * n + g] =
                dfloat(P.pp[((size_t)(PP_PX + x) * PIMD_MAXPP + k) * n + g] - S.xyz[3 * sb + x]);
    }
}

void launch_pair_dfloat(const Pairs& P, const Shells& S, dfloat* ppd, dfloat* abd, cudaStream_t st)
{
    if (P.n == 0) return;
    pair_dfloat_kernel<<<(P.n + 127) / 128, 128, 0, st>>>(P, S, ppd, abd);
}

__global__ void to_float_kernel(const double* src, float* dst, long long n)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = (float)src[i];
}

void launch_to_float(const double* src, float* dst, long long n, cudaStream_t st)
{
    if (n <= 0) return;
    to_float_kernel<<<256, 256, 0, st>>>(src, dst, n);
}

}  // namespace pimd
