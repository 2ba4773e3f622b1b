// Shell-quartet ERI kernels: Coulomb/exchange (Fock) build, Schwarz factors
// and the two-electron part of the analytic RHF gradient.
//
// One thread, or several lanes of a warp where quartets are few, evaluates one
// contracted shell quartet (ab|cd) of one replica, in FP64, float-float
// (dfloat.cuh) or FP32: the primitive loop runs the generated Obara-Saika
// vertical recursion into contracted [e0|f0] accumulators, then the generated
// Head-Gordon-Pople horizontal recursion gives the Cartesian block, which is turned into real
// spherical d functions and contracted with the density on the fly.
// A block shares one bra pair (staged in shared memory) and walks a tile of
// 32, 64 or 128 ket pairs of the same class (the width is chosen per class pair
// by the autotuner), so the code path is uniform across
// the block. Every replica of the call is covered by the same launch.
//
// Quartets are the canonical ones (a >= b, c >= d, ab >= cd); each is
// scattered to its 8 permutations with weight f = 1/|stabiliser| into a
// non-symmetric G' with F = h + G' + G'^T, where (per element)
//   G'_ab += 2f D_cd v,  G'_cd += 2f D_ab v,
//   G'_ac -= f/2 D_bd v, G'_bc -= f/2 D_ad v, G'_ad -= f/2 D_bc v, G'_bd -= f/2 D_ac v,
// which reproduces F = h + J - K/2 with J_mn = sum D_ls (mn|ls) and
// K_mn = sum D_ls (ml|ns) for a symmetric density.
#pragma once
#include <type_traits>

#include "boys.cuh"
#include "pimd_dev.cuh"

namespace pimd {

// Float-float Fock kernels, by the operations of the class's recursion: above
// the first, the packed recursion (two nodes to an instruction; (dp|ps) 17.7 ->
// 15.3 ms, (dp|dp) 62.5 -> 36.9 for 8 (H2O)8 beads, but (pp|ps), below it, 12.3
// -> 13.0: the packed form costs registers and its gain is code size); above
// the second, the horizontal recursion, transform and J/K contraction in FP64
// ((dp|ps) 15.3 -> 13.3 ms, (dp|ds) 19.3 -> 16.7): the FP64 pipe is idle, and
// their code leaves the instruction caches to the primitive loop.
constexpr int DF_PACKED_MIN_FLOPS = 300, DF_TAIL64_MIN_FLOPS = 500;
// their primitive cutoff as a fraction of the FP64 kernels': what it keeps more
// outweighs the float-float rounding in the error of the Fock matrix (kDfTau
// has the figures), for 1% of the time
constexpr double DF_TAU_PRIM = 0.8;

constexpr double kSqrt3 = 1.7320508075688772935;

// in[N0][ncart(L)][N2] -> out[N0][nsph(L)][N2]; spherical d order m = -2..2:
// sqrt3 xy, sqrt3 yz, zz - (xx + yy)/2, sqrt3 xz, sqrt3/2 (xx - yy)
template <int N0, int L, int N2, typename T>
__device__ __forceinline__ void sph_index(const T* __restrict__ in, T* __restrict__ out)
{
    if constexpr (L < 2) {
#pragma unroll
        for (int i = 0; i < N0 * ncart(L) * N2; i++) out[i] = in[i];
    } else {
#pragma unroll
        for (int i0 = 0; i0 < N0; i0++)
#pragma unroll
            for (int i2 = 0; i2 < N2; i2++) {
                const T* s = in + i0 * 6 * N2 + i2;
                T* d = out + i0 * 5 * N2 + i2;
                const T xx = s[0], xy = s[N2], xz = s[2 * N2], yy = s[3 * N2], yz = s[4 * N2], zz = s[5 * N2];
                d[0] = T(kSqrt3) * xy;
                d[N2] = T(kSqrt3) * yz;
                d[2 * N2] = zz - T(0.5) * (xx + yy);
                d[3 * N2] = T(kSqrt3) * xz;
                d[4 * N2] = T(0.5 * kSqrt3) * (xx - yy);
            }
    }
}

// transpose of sph_index: in[N0][nsph(L)][N2] -> out[N0][ncart(L)][N2]
template <int N0, int L, int N2, typename T>
__device__ __forceinline__ void sph_index_t(const T* __restrict__ in, T* __restrict__ out)
{
    if constexpr (L < 2) {
#pragma unroll
        for (int i = 0; i < N0 * ncart(L) * N2; i++) out[i] = in[i];
    } else {
#pragma unroll
        for (int i0 = 0; i0 < N0; i0++)
#pragma unroll
            for (int i2 = 0; i2 < N2; i2++) {
                const T* s = in + i0 * 5 * N2 + i2;
                T* d = out + i0 * 6 * N2 + i2;
                const T m2 = s[0], m1 = s[N2], m0 = s[2 * N2], p1 = s[3 * N2], p2 = s[4 * N2];
                d[0] = T(-0.5) * m0 + T(0.5 * kSqrt3) * p2;
                d[N2] = T(kSqrt3) * m2;
                d[2 * N2] = T(kSqrt3) * p1;
                d[3 * N2] = T(-0.5) * m0 - T(0.5 * kSqrt3) * p2;
                d[4 * N2] = T(kSqrt3) * m1;
                d[5 * N2] = m0;
            }
    }
}

// Cartesian (ab|cd) block -> spherical block
template <int LA, int LB, int LC, int LD, typename T>
__device__ __forceinline__ void cart_to_sph4(T* __restrict__ buf, T* __restrict__ tmp)
{
    constexpr int ca = ncart(LA), cb = ncart(LB), cc = ncart(LC), cd = ncart(LD);
    constexpr int sa = nsph(LA), sb = nsph(LB), sc = nsph(LC);
    sph_index<1, LA, cb * cc * cd>(buf, tmp);
    sph_index<sa, LB, cc * cd>(tmp, buf);
    sph_index<sa * sb, LC, cd>(buf, tmp);
    sph_index<sa * sb * sc, LD, 1>(tmp, buf);
}

template <int LA, int LB, int LC, int LD, typename T>
__device__ __forceinline__ void sph_to_cart4_t(T* __restrict__ buf, T* __restrict__ tmp)
{
    constexpr int ca = ncart(LA), cb = ncart(LB), cc = ncart(LC);
    constexpr int sb = nsph(LB), sc = nsph(LC), sd = nsph(LD);
    sph_index_t<1, LA, sb * sc * sd>(buf, tmp);
    sph_index_t<ca, LB, sc * sd>(tmp, buf);
    sph_index_t<ca * cb, LC, sd>(buf, tmp);
    sph_index_t<ca * cb * cc, LD, 1>(tmp, buf);
}

// Per-primitive-quartet quantities of the Obara-Saika recursion.
template <typename R>
struct PrimQ {
    R PA[3], WP[3], QC[3], WQ[3];
    R o2p, o2pr, o2q, o2qr, o2pq, T, theta;
};
typedef PrimQ<double> PrimQuartet;

__device__ __forceinline__ float rsqrt_r(float x) { return rsqrtf(x); }

// bra/ket: the first PP_NERI primitive-pair fields (p, P, K, P - A, 1/(2p), 1/(2p^2))
template <typename R>
__device__ __forceinline__ void prim_quartet(const R* bra, const R* ket, PrimQ<R>& g)
{
    const R p = bra[PP_P], q = ket[PP_P];
    const R rs = rsqrt_r(p + q);
    const R ipq = rs * rs;
    const R qi = q * ipq, pi = p * ipq;
    const R rho = p * qi;
    const R PQx = bra[PP_PX] - ket[PP_PX], PQy = bra[PP_PY] - ket[PP_PY], PQz = bra[PP_PZ] - ket[PP_PZ];
    // W - P = -q/(p+q) (P - Q), W - Q = p/(p+q) (P - Q)
    g.WP[0] = -qi * PQx;
    g.WP[1] = -qi * PQy;
    g.WP[2] = -qi * PQz;
    g.WQ[0] = pi * PQx;
    g.WQ[1] = pi * PQy;
    g.WQ[2] = pi * PQz;
    g.PA[0] = bra[PP_PAX];
    g.PA[1] = bra[PP_PAY];
    g.PA[2] = bra[PP_PAZ];
    g.QC[0] = ket[PP_PAX];
    g.QC[1] = ket[PP_PAY];
    g.QC[2] = ket[PP_PAZ];
    g.T = rho * fma(PQx, PQx, fma(PQy, PQy, PQz * PQz));
    g.o2p = bra[PP_O2P];
    g.o2pr = rho * bra[PP_O2PP];
    g.o2q = ket[PP_O2P];
    g.o2qr = rho * ket[PP_O2PP];
    g.o2pq = R(0.5) * ipq;
    g.theta = bra[PP_K] * ket[PP_K] * rs;
}

// How the float-float kernels form P - Q of a quartet: as (P - X) - (Q - Y) +
// (X - Y) with X the bra centre A or B and Y the ket centre C or D, on the same
// atom where the quartet has such a pair. The product centres of two tight
// primitives can then be as close as they are (the integral varies over
// 1/sqrt(rho)), where a difference of coordinates, or of a centre other than the
// near one, would leave 2^-48 of a bond length or of the molecule's size. X - Y
// of two atoms is the FP64 difference, made a float-float afterwards: of the
// coordinates as float-floats it would lose 2^-48 of the distance from the
// origin, 32 times what FP64 does.
struct DfCentres {
    int bra, ket;     // first of the three fields P - X: PP_PAX or PP_PBX
    dfloat XY[3];
    __device__ __forceinline__ DfCentres(const Shells& S, int sa, int sb, int sc, int sd)
    {
        const int a = S.atom[sa], b = S.atom[sb], c = S.atom[sc], d = S.atom[sd];
        bra = a == c || a == d || (b != c && b != d) ? PP_PAX : PP_PBX;
        ket = (bra == PP_PAX ? a : b) == d && (bra == PP_PAX ? a : b) != c ? PP_PBX : PP_PAX;
        const int x = bra == PP_PAX ? sa : sb, y = ket == PP_PAX ? sc : sd;
#pragma unroll
        for (int k = 0; k < 3; k++) XY[k] = dfloat(__ldg(S.xyz + 3 * x + k) - __ldg(S.xyz + 3 * y + k));
    }
    // X - Y - (Q - Y) of ket primitive j of pair cd
    __device__ __forceinline__ void ket_part(const Pairs& P, int cd, int j, dfloat aq[3]) const
    {
#pragma unroll
        for (int k = 0; k < 3; k++)
            aq[k] = XY[k] - ldg(P.ppd + ((size_t)(ket + k) * PIMD_MAXPP + j) * P.n + cd);
    }
};

// The same from float-float pair data: bra primitive i of sbra, aq from
// DfCentres::ket_part.
__device__ __forceinline__ void prim_quartet(const dfloat (*sbra)[PIMD_MAXPP], int i, const DfCentres& ctr,
                                             const dfloat* ket, const dfloat* aq, PrimQ<dfloat>& g)
{
    const dfloat p = sbra[PP_P][i], q = ket[PP_P];
    const dfloat rs = rsqrt_r(p + q);
    const dfloat ipq = rs * rs;
    const dfloat qi = q * ipq, pi = p * ipq;
    const dfloat rho = p * qi;
    dfloat PQ[3];
#pragma unroll
    for (int x = 0; x < 3; x++) {
        g.PA[x] = sbra[PP_PAX + x][i];
        g.QC[x] = ket[PP_PAX + x];
        PQ[x] = aq[x] + sbra[ctr.bra + x][i];
        g.WP[x] = -(qi * PQ[x]);
        g.WQ[x] = pi * PQ[x];
    }
    g.T = renorm(rho * fma(PQ[0], PQ[0], fma(PQ[1], PQ[1], PQ[2] * PQ[2])));
    g.o2p = sbra[PP_O2P][i];
    g.o2pr = rho * sbra[PP_O2PP][i];
    g.o2q = ket[PP_O2P];
    g.o2qr = rho * ket[PP_O2PP];
    g.o2pq = scale2(ipq, 0.5f);
    g.theta = sbra[PP_K][i] * ket[PP_K] * rs;
}

// rows of a kernel's shared bra data
template <typename R>
constexpr int bra_rows(int n) { return std::is_same<R, dfloat>::value ? (int)PPD_NF : n; }

__device__ __forceinline__ double shfl_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ float shfl_xor(float v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ dfloat shfl_xor(dfloat v, int o)
{
    return dfloat(__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o));
}

// sum over the warp, and c v as a double (c a power of two times a sign)
__device__ __forceinline__ dfloat warp_sum_any(dfloat v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += shfl_xor(v, o);
    return v;
}
__device__ __forceinline__ double warp_sum_any(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double scaled(dfloat v, double c) { return (double)scale2(v, (float)c); }
__device__ __forceinline__ double scaled(double v, double c) { return c * v; }
__device__ __forceinline__ double scaled(float v, double c) { return c * (double)v; }

// J'_ab of a tile: every lane of the warp holds a quartet with the same bra
// pair (ab), so the bra-side Coulomb block sum_cd 2f D_cd (ab|cd) is summed
// over the warp with shuffles and added to G' with one atomic per element
// (lanes without a quartet contribute zero; all 32 lanes must call this).
template <int LA, int LB, int LC, int LD, typename R>
__device__ __forceinline__ void bra_coulomb_warp(const R* __restrict__ I, double f, bool work, int fa, int fb,
                                                 int fc, int fd, int N, const R* __restrict__ D,
                                                 double* __restrict__ G, double fxs)
{
    constexpr int na = nsph(LA), nb = nsph(LB), nc = nsph(LC), nd = nsph(LD);
    R Dcd[nc * nd];
#pragma unroll
    for (int i = 0; i < nc; i++)
#pragma unroll
        for (int j = 0; j < nd; j++) Dcd[i * nd + j] = work ? ldg(D + (size_t)(fc + i) * N + fd + j) : R(0);
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int a = 0; a < na; a++) {
#pragma unroll
        for (int b = 0; b < nb; b++) {
            R s = R(0);
#pragma unroll
            for (int c = 0; c < nc; c++)
#pragma unroll
                for (int d = 0; d < nd; d++) s += Dcd[c * nd + d] * I[((a * nb + b) * nc + c) * nd + d];
            double v;
            if constexpr (std::is_same<R, dfloat>::value) {
                // (the weight is a power of two: exact on both parts)
                v = (double)warp_sum_any(work ? scale2(s, (float)(2.0 * f)) : R(0));
            } else {
                v = warp_sum_any(work ? 2.0 * f * (double)s : 0.0);
            }
            if (lane == 0 && v != 0.0) det_add(G + (size_t)(fa + a) * N + fb + b, v, fxs);
        }
    }
}

// Contract a spherical block with the density and scatter into G' (the
// contraction in the block's precision R, the accumulation in FP64): J'_cd
// and the four exchange blocks; with bra_j, also J'_ab (else the caller adds
// it with bra_coulomb_warp).
template <int LA, int LB, int LC, int LD, typename R>
__device__ __forceinline__ void scatter_jk(const R* __restrict__ I, double f, int fa, int fb, int fc, int fd,
                                           int N, const R* __restrict__ D, double* __restrict__ G, double fxs,
                                           bool bra_j = true)
{
    constexpr int na = nsph(LA), nb = nsph(LB), nc = nsph(LC), nd = nsph(LD);
    R Dab[na * nb], Dcd[nc * nd], Dac[na * nc], Dad[na * nd], Dbc[nb * nc], Dbd[nb * nd];
#pragma unroll
    for (int i = 0; i < na; i++)
#pragma unroll
        for (int j = 0; j < nb; j++) Dab[i * nb + j] = ldg(D + (size_t)(fa + i) * N + fb + j);
#pragma unroll
    for (int i = 0; i < nc; i++)
#pragma unroll
        for (int j = 0; j < nd; j++) Dcd[i * nd + j] = ldg(D + (size_t)(fc + i) * N + fd + j);
#pragma unroll
    for (int i = 0; i < na; i++)
#pragma unroll
        for (int j = 0; j < nc; j++) Dac[i * nc + j] = ldg(D + (size_t)(fa + i) * N + fc + j);
#pragma unroll
    for (int i = 0; i < na; i++)
#pragma unroll
        for (int j = 0; j < nd; j++) Dad[i * nd + j] = ldg(D + (size_t)(fa + i) * N + fd + j);
#pragma unroll
    for (int i = 0; i < nb; i++)
#pragma unroll
        for (int j = 0; j < nc; j++) Dbc[i * nc + j] = ldg(D + (size_t)(fb + i) * N + fc + j);
#pragma unroll
    for (int i = 0; i < nb; i++)
#pragma unroll
        for (int j = 0; j < nd; j++) Dbd[i * nd + j] = ldg(D + (size_t)(fb + i) * N + fd + j);

    // J'_ab (rows of the bra)
    if (bra_j) {
#pragma unroll
        for (int a = 0; a < na; a++) {
#pragma unroll
            for (int b = 0; b < nb; b++) {
                R s = R(0);
#pragma unroll
                for (int c = 0; c < nc; c++)
#pragma unroll
                    for (int d = 0; d < nd; d++) s += Dcd[c * nd + d] * I[((a * nb + b) * nc + c) * nd + d];
                det_add(G + (size_t)(fa + a) * N + fb + b, scaled(s, 2.0 * f), fxs);
            }
        }
    }
#pragma unroll
    for (int c = 0; c < nc; c++)
#pragma unroll
        for (int d = 0; d < nd; d++) {
            R s = R(0);
#pragma unroll
            for (int a = 0; a < na; a++)
#pragma unroll
                for (int b = 0; b < nb; b++) s += Dab[a * nb + b] * I[((a * nb + b) * nc + c) * nd + d];
            det_add(G + (size_t)(fc + c) * N + fd + d, scaled(s, 2.0 * f), fxs);
        }
#pragma unroll
    for (int a = 0; a < na; a++)
#pragma unroll
        for (int c = 0; c < nc; c++) {
            R s = R(0);
#pragma unroll
            for (int b = 0; b < nb; b++)
#pragma unroll
                for (int d = 0; d < nd; d++) s += Dbd[b * nd + d] * I[((a * nb + b) * nc + c) * nd + d];
            det_add(G + (size_t)(fa + a) * N + fc + c, scaled(s, -0.5 * f), fxs);
        }
#pragma unroll
    for (int b = 0; b < nb; b++)
#pragma unroll
        for (int c = 0; c < nc; c++) {
            R s = R(0);
#pragma unroll
            for (int a = 0; a < na; a++)
#pragma unroll
                for (int d = 0; d < nd; d++) s += Dad[a * nd + d] * I[((a * nb + b) * nc + c) * nd + d];
            det_add(G + (size_t)(fb + b) * N + fc + c, scaled(s, -0.5 * f), fxs);
        }
#pragma unroll
    for (int a = 0; a < na; a++)
#pragma unroll
        for (int d = 0; d < nd; d++) {
            R s = R(0);
#pragma unroll
            for (int b = 0; b < nb; b++)
#pragma unroll
                for (int c = 0; c < nc; c++) s += Dbc[b * nc + c] * I[((a * nb + b) * nc + c) * nd + d];
            det_add(G + (size_t)(fa + a) * N + fd + d, scaled(s, -0.5 * f), fxs);
        }
#pragma unroll
    for (int b = 0; b < nb; b++)
#pragma unroll
        for (int d = 0; d < nd; d++) {
            R s = R(0);
#pragma unroll
            for (int a = 0; a < na; a++)
#pragma unroll
                for (int c = 0; c < nc; c++) s += Dac[a * nc + c] * I[((a * nb + b) * nc + c) * nd + d];
            det_add(G + (size_t)(fb + b) * N + fd + d, scaled(s, -0.5 * f), fxs);
        }
}

// first nf primitive-pair fields of pair g, primitive pair k
__device__ __forceinline__ void load_ppn(const Pairs& P, int g, int k, double* out, int nf)
{
    const size_t n = P.n;
#pragma unroll
    for (int f = 0; f < nf; f++) out[f] = __ldg(P.pp + ((size_t)f * PIMD_MAXPP + k) * n + g);
}
__device__ __forceinline__ void load_ppn(const Pairs& P, int g, int k, float* out, int nf)
{
    const size_t n = P.n;
#pragma unroll
    for (int f = 0; f < nf; f++) out[f] = __ldg(P.ppf + ((size_t)f * PIMD_MAXPP + k) * n + g);
}
__device__ __forceinline__ void load_ppn(const Pairs& P, int g, int k, dfloat* out, int nf)
{
    const size_t n = P.n;
#pragma unroll
    for (int f = 0; f < nf; f++) out[f] = ldg(P.ppd + ((size_t)f * PIMD_MAXPP + k) * n + g);
}
__device__ __forceinline__ const dfloat* pp_base(const Pairs& P, dfloat) { return P.ppd; }
__device__ __forceinline__ const double* pp_base(const Pairs& P, double) { return P.pp; }
__device__ __forceinline__ const float* pp_base(const Pairs& P, float) { return P.ppf; }

// contracted Cartesian block of one quartet via the generated recursion.
// Primitive screening: primitive quartet (i|j) is skipped when
// qp_i qp_j < qthr (qthr = the primitive cutoff over the quartet's density
// bound; qthr <= 0 keeps every primitive); both primitive lists are in
// descending order of qp, so the quartets that survive form a staircase: for
// ket primitive j the bra primitives i < imax(j), imax non-increasing. The
// loop walks that staircase as one flat sequence of `total` primitive
// quartets, and runs `kmax` iterations (kmax >= total, the longest sequence
// of the warp), so that a warp executes the recursion once per position of
// its longest lane instead of once per primitive quartet that any lane needs.
// Returns the number of primitive quartets evaluated.
__device__ __forceinline__ int stair_width(const float* sqp, int nbra, float qj, float qthr)
{
    int n = 0;
    while (n < nbra && sqp[n] * qj >= qthr) n++;
    return n;
}

__device__ __forceinline__ int stair_total(const float* sqp, int nbra, const Pairs& P, int cd, float qthr)
{
    const int nket = P.npp[cd];
    if (qthr <= 0.0f) return nbra * nket;
    int total = 0;
    for (int j = 0; j < nket; j++) {
        const int w = stair_width(sqp, nbra, __ldg(P.qp + (size_t)j * P.n + cd), qthr);
        if (w == 0) break;
        total += w;
    }
    return total;
}

// S lanes of a warp (S a power of two, sub = 0..S-1 of this one) share a
// quartet: each takes every S-th position of the sequence, and the
// contracted accumulators are summed over them before the horizontal
// recursion. Every lane of the warp calls this (total = 0: no quartet; cd then
// any pair); kmax: the longest sequence of the warp.
// Float-float classes: which ones use the packed recursion, and which hand the
// contracted accumulators to FP64 for the horizontal recursion, the spherical
// transform and the J/K contraction (Tail: the type of those).
template <class C, typename R>
struct DfClass {
    static constexpr bool df = std::is_same<R, dfloat>::value;
    static constexpr bool packed = df && C::VRR_FLOPS > DF_PACKED_MIN_FLOPS;
    typedef typename std::conditional<df && (C::VRR_FLOPS > DF_TAIL64_MIN_FLOPS), double, R>::type Tail;
};
template <typename R>
__device__ __forceinline__ R to_tail(R v, R) { return v; }
__device__ __forceinline__ double to_tail(dfloat v, double) { return (double)v; }

template <class C, typename R, typename T>
__device__ __forceinline__ void quartet_cart(const R (*sbra)[PIMD_MAXPP], const float* sqp, int nbra, const Pairs& P,
                                             int cd, const T AB[3], const T CD[3], const DfCentres* ctr,
                                             const R* __restrict__ boys, float qthr, int total, int kmax, int S,
                                             int sub, T* cart)
{
    constexpr bool DF = std::is_same<R, dfloat>::value, PACKED = DfClass<C, R>::packed;
    // (the float-float recursion is packed, two nodes to an operation)
    R acc[C::NE * C::NF];
    dfloat2 acc2[PACKED ? C::N2 : 1];
    if constexpr (PACKED) {
#pragma unroll
        for (int i = 0; i < C::N2; i++) acc2[i] = dfloat2(make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f));
    } else {
#pragma unroll
        for (int i = 0; i < C::NE * C::NF; i++) acc[i] = R(0);
    }
    // position `pos` of the sequence = bra primitive i of ket primitive j,
    // whose row is w long
    int i = sub, j = 0, jl = -1;
    int w = total > 0 ? (qthr > 0.0f ? stair_width(sqp, nbra, __ldg(P.qp + cd), qthr) : nbra) : 0;
    R ket[PP_NERI], aq[3];
    for (int k = 0; k < kmax; k += S) {
        if (k + sub < total) {
            while (i >= w) {
                i -= w;
                j++;
                if (qthr > 0.0f) w = stair_width(sqp, nbra, __ldg(P.qp + (size_t)j * P.n + cd), qthr);
            }
            if (j != jl) {
                load_ppn(P, cd, j, ket, PP_NERI);
                jl = j;
                if constexpr (DF) ctr->ket_part(P, cd, j, aq);
            }
            PrimQ<R> g;
            if constexpr (DF) {
                prim_quartet(sbra, i, *ctr, ket, aq, g);
            } else {
                R bra[PP_NERI];
#pragma unroll
                for (int f = 0; f < PP_NERI; f++) bra[f] = sbra[f][i];
                prim_quartet<R>(bra, ket, g);
            }
            R F[C::L + 1];
            boys_eval<C::L>(g.T, boys, g.theta, F);
            if constexpr (PACKED) {
                // what a long recursion reads many times, with normalised low parts
#pragma unroll
                for (int m = 0; m <= C::L; m++) F[m] = renorm(F[m]);
#pragma unroll
                for (int x = 0; x < 3; x++) {
                    g.WP[x] = renorm(g.WP[x]);
                    g.WQ[x] = renorm(g.WQ[x]);
                }
                g.o2pr = renorm(g.o2pr);
                g.o2qr = renorm(g.o2qr);
                g.o2pq = renorm(g.o2pq);
                C::vrr2(F, g, acc2);
            }
            else
                C::template vrr<R>(F, g.PA[0], g.PA[1], g.PA[2], g.WP[0], g.WP[1], g.WP[2], g.QC[0], g.QC[1], g.QC[2],
                                   g.WQ[0], g.WQ[1], g.WQ[2], g.o2p, g.o2pr, g.o2q, g.o2qr, g.o2pq, acc);
            i += S;
        }
    }
    if constexpr (PACKED) C::vrr2_unpack(acc2, acc);
    for (int o = 1; o < S; o <<= 1)
#pragma unroll
        for (int e = 0; e < C::NE * C::NF; e++) acc[e] += shfl_xor(acc[e], o);
    T acct[C::NE * C::NF];
#pragma unroll
    for (int e = 0; e < C::NE * C::NF; e++) acct[e] = to_tail(acc[e], T());
    if (sub == 0) C::template hrr<T>(acct, AB[0], AB[1], AB[2], CD[0], CD[1], CD[2], cart);
}

// Blocks per tile of the straight-line kernels (gridDim.y): a block takes every
// gridDim.y-th of the tile's quartets and, where few are left to it, several
// lanes per quartet, so a small batch's primitive loops are spread over the
// chip instead of running 81 recursions deep on a few warps. Two where a class
// has fewer tiles than the chip holds blocks (2 per SM); its launch runs beside
// those of the other classes, and more blocks repeat the set-up and the serial
// end of a quartet for ever fewer of them: one (H2O)8 bead's Fock builds 398 /
// 364 / 386 ms with 1 / 2 / up to 8 blocks per tile below 152 / 304 / 608 tiles,
// 4 dimers' 55 / 59 / 72, ragged images' 173 / 164 / 186.
// With the float-float kernels and the lane sharing: the Fock build of one water
// molecule 18.8 -> 6.3 ms, the forces of 4 minimal-basis dimers 37.3 -> 12.5 ms,
// of one (H2O)8 bead 1196 -> 843 ms.
inline int jk_blocks_per_tile(int ntiles) { return ntiles < 2 * 152 ? 2 : 1; }

// tau_prim: primitive quartets whose bound qp_i qp_j (density bound) is below
// it are skipped (0 keeps every primitive quartet). fxs > 0: G' accumulated as
// fixed-point integers (det_add).
template <class C, typename R>
__global__ void __launch_bounds__(128) jk_kernel(Pairs P, Shells S_, Reps R_, const Tile* __restrict__ tiles,
                                                 const typename DfClass<C, R>::Tail* __restrict__ Dall,
                                                 double* __restrict__ Gall,
                                                 const R* __restrict__ boys, double tau_lo, double tau_hi,
                                                 const double* __restrict__ Dsh, unsigned long long* __restrict__ cnt,
                                                 double tau_prim, double fxs)
{
    typedef typename DfClass<C, R>::Tail T;
    constexpr int ROWS = bra_rows<R>(PP_NERI);
    __shared__ R sbra[ROWS][PIMD_MAXPP];
    __shared__ float sqp[PIMD_MAXPP];
    const Tile t = tiles[blockIdx.x];
    if (!R_.active[t.rep]) return;
    const int ab = t.ab;
    for (int e = threadIdx.x; e < ROWS * PIMD_MAXPP; e += blockDim.x) {
        const int f = e / PIMD_MAXPP, k = e % PIMD_MAXPP;
        sbra[f][k] = pp_base(P, R())[((size_t)f * PIMD_MAXPP + k) * P.n + ab];
    }
    if (threadIdx.x < PIMD_MAXPP) sqp[threadIdx.x] = P.qp[(size_t)threadIdx.x * P.n + ab];
    __syncthreads();
    const int r = t.rep;
    const int nbra = P.npp[ab];
    // screening of ket pair c0 + k: density-weighted Schwarz bound (every
    // contribution of the quartet to G' is at most 2 |(ab|cd)| times one of
    // the six density blocks) and the primitive cutoff over that bound
    auto screen = [&](int k, int& cd, int& sc, int& sd, float& qthr) -> bool {
        cd = t.c0 + k;
        sc = sd = 0;
        qthr = 0.0f;
        if (cd >= t.c1) return false;
        const int sa = P.sa[ab], sb = P.sb[ab];
        sc = P.sa[cd];
        sd = P.sb[cd];
        const double dq = fmax(fmax(fmax(shell_bound(R_, Dsh, r, sa, sb), shell_bound(R_, Dsh, r, sc, sd)),
                                    fmax(shell_bound(R_, Dsh, r, sa, sc), shell_bound(R_, Dsh, r, sa, sd))),
                               fmax(shell_bound(R_, Dsh, r, sb, sc), shell_bound(R_, Dsh, r, sb, sd)));
        const double bound = P.Q[ab] * P.Q[cd] * dq;
        qthr = (float)(tau_prim / dq);
        return bound >= tau_lo && bound < tau_hi;
    };
    int cd, sc, sd;
    float qthr;
    bool work = screen(threadIdx.x, cd, sc, sd, qthr);
    const int tid = threadIdx.x, bd = blockDim.x;
    // quartets of the tile that are left, and this block's share of them
    const int nwork = __syncthreads_count(work);
    const int mine = (nwork - (int)blockIdx.y + (int)gridDim.y - 1) / (int)gridDim.y;
    if (mine <= 0) return;
    // Lanes stop their primitive loops at their own cutoff, and a warp issues
    // for all its lanes: the tile's quartets are regrouped by the number of
    // primitive quartets that survive (descending, bitonic sort over the
    // block; the ones screened out last), so that a warp holds quartets of
    // similar length. Lanes without a quartet of their own are given to the
    // others, S to a quartet; the FP32 quartets keep one lane each, and with it
    // the order of their sums.
    __shared__ int skey[128], sidx[128];
    skey[tid] = work ? stair_total(sqp, nbra, P, cd, qthr) : -1;
    sidx[tid] = tid;
    __syncthreads();
    for (int k = 2; k <= bd; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            const int o = tid ^ j;
            if (o > tid) {
                const bool desc = (tid & k) == 0;
                const int a = skey[tid], b = skey[o];
                if (desc ? a < b : a > b) {
                    skey[tid] = b;
                    skey[o] = a;
                    const int x = sidx[tid];
                    sidx[tid] = sidx[o];
                    sidx[o] = x;
                }
            }
            __syncthreads();
        }
    int S = 1;
    if constexpr (!std::is_same<R, float>::value)
        while (S < 32 && 2 * S * mine <= bd) S *= 2;
    const int item = tid / S, sub = tid % S;
    work = item < mine && screen(sidx[blockIdx.y + item * gridDim.y], cd, sc, sd, qthr);
    const int sa = P.sa[ab], sb = P.sb[ab];
    // a warp with no quartet left leaves; otherwise every lane stays for the
    // sums over lanes (the block's warps share the bra pair)
    if (__all_sync(0xffffffffu, !work)) return;
    constexpr int NCART = ncart(C::LA) * ncart(C::LB) * ncart(C::LC) * ncart(C::LD);
    T cart[NCART], tmp[NCART];
    const int total = work ? stair_total(sqp, nbra, P, cd, qthr) : 0;
    const int kmax = __reduce_max_sync(0xffffffffu, (unsigned)total);
    T AB[3], CD[3];
    if (work) {
#pragma unroll
        for (int x = 0; x < 3; x++) {
            if constexpr (std::is_same<T, dfloat>::value) {
                AB[x] = ldg(P.abd + (size_t)x * P.n + ab);
                CD[x] = ldg(P.abd + (size_t)x * P.n + cd);
            } else {
                AB[x] = T(S_.xyz[3 * sa + x] - S_.xyz[3 * sb + x]);
                CD[x] = T(S_.xyz[3 * sc + x] - S_.xyz[3 * sd + x]);
            }
        }
    }
    if constexpr (DfClass<C, R>::df) {
        const DfCentres ctr(S_, sa, sb, work ? sc : sa, work ? sd : sb);
        quartet_cart<C, R, T>(sbra, sqp, nbra, P, cd, AB, CD, &ctr, boys, qthr, total, kmax, S, sub, cart);
    } else {
        quartet_cart<C, R, T>(sbra, sqp, nbra, P, cd, AB, CD, nullptr, boys, qthr, total, kmax, S, sub, cart);
    }
    work = work && sub == 0;
    double f = 0.0;
    if (work) {
        cart_to_sph4<C::LA, C::LB, C::LC, C::LD>(cart, tmp);
        f = 1.0;
        if (sa == sb) f *= 0.5;
        if (sc == sd) f *= 0.5;
        if (ab == cd) f *= 0.5;
    }
    const unsigned nq = __reduce_add_sync(0xffffffffu, work ? 1u : 0u);
    const unsigned np = __reduce_add_sync(0xffffffffu, work ? (unsigned)total : 0u);
    if ((threadIdx.x & 31) == 0 && nq) {
        atomicAdd(cnt, (unsigned long long)nq);
        atomicAdd(cnt + 1, (unsigned long long)np);
        atomicAdd(R_.qrep + 2 * r + (sizeof(R) == 4 ? 1 : 0), (unsigned long long)nq);
    }
    const int N = R_.nbf[r];
    const size_t off = R_.moff[r];
    bra_coulomb_warp<C::LA, C::LB, C::LC, C::LD, T>(cart, f, work, S_.bf[P.sa[ab]], S_.bf[P.sb[ab]], S_.bf[sc],
                                                     S_.bf[sd], N, Dall + off, Gall + off, fxs);
    if (work)
        scatter_jk<C::LA, C::LB, C::LC, C::LD, T>(cart, f, S_.bf[sa], S_.bf[sb], S_.bf[sc], S_.bf[sd], N, Dall + off,
                                                  Gall + off, fxs, false);
}

// Contracted Cartesian block (ab|ab) of the primitive quartets first, first +
// stride, ... < np * np of one pair (primitive i of the bra, j of the ket at
// j * np + i), spherical: the recursions and the transform are linear, so the
// blocks of a pair's threads add up to the whole.
template <class C>
__device__ __forceinline__ void pair_block(const Pairs& P, const double* pp, int ab, const double A[3],
                                           const double B[3], int np, int first, int last, int stride,
                                           const double* __restrict__ boys, double* cart)
{
    const size_t n = P.n;
    double acc[C::NE * C::NF];
#pragma unroll
    for (int i = 0; i < C::NE * C::NF; i++) acc[i] = 0.0;
    for (int q = first; q < last; q += stride) {
        double bra[PP_NERI], ket[PP_NERI];
#pragma unroll
        for (int f = 0; f < PP_NERI; f++) {
            bra[f] = pp[((size_t)f * PIMD_MAXPP + q % np) * n + ab];
            ket[f] = pp[((size_t)f * PIMD_MAXPP + q / np) * n + ab];
        }
        PrimQ<double> g;
        prim_quartet<double>(bra, ket, g);
        double F[C::L + 1];
        boys_eval<C::L>(g.T, boys, g.theta, F);
        C::template vrr<double>(F, g.PA[0], g.PA[1], g.PA[2], g.WP[0], g.WP[1], g.WP[2], g.QC[0], g.QC[1], g.QC[2],
                                g.WQ[0], g.WQ[1], g.WQ[2], g.o2p, g.o2pr, g.o2q, g.o2qr, g.o2pq, acc);
    }
    constexpr int NCART = ncart(C::LA) * ncart(C::LB) * ncart(C::LC) * ncart(C::LD);
    double tmp[NCART];
    C::template hrr<double>(acc, A[0] - B[0], A[1] - B[1], A[2] - B[2], A[0] - B[0], A[1] - B[1], A[2] - B[2], cart);
    cart_to_sph4<C::LA, C::LB, C::LC, C::LD>(cart, tmp);
}

// the density the float-float kernel of class C contracts with
template <class C>
static const typename DfClass<C, dfloat>::Tail* tail_density(const double* D, const dfloat* Dd)
{
    if constexpr (std::is_same<typename DfClass<C, dfloat>::Tail, double>::value)
        return D;
    else
        return Dd;
}

// Schwarz factors: Q_ab = sqrt(max over functions of (mn|mn)), one block per
// pair. The pair's primitive quartets (up to 81) are spread over the block's
// threads, each with its own contracted block, and only the diagonal elements
// (mn|mn) are summed over the block. Bound by the latency of one thread's
// FP64 chain ((dd|dd): about 9000 FMAs per primitive quartet), not by
// throughput: one thread per pair, as before, ran 81 of them one after
// another ((dd|dd) of one (H2O)8 bead, 36 pairs: 57 ms).
// A Fock build of one water molecule (24 functions), most of it this set-up:
// 91.6 -> 18.9 ms with this kernel and the next.
// blockDim.x = SCHWARZ_WIDE threads (one primitive quartet each) or one warp.
constexpr int SCHWARZ_WIDE = 96;

template <class C>
__global__ void __launch_bounds__(SCHWARZ_WIDE) schwarz_kernel(Pairs P, Shells S, const int* __restrict__ list, int n,
                                                               const double* __restrict__ boys,
                                                               double* __restrict__ Qout)
{
    constexpr int na = nsph(C::LA), nb = nsph(C::LB);
    __shared__ double s_diag[SCHWARZ_WIDE / 32][na * nb];
    const int ab = list[blockIdx.x];
    const int sa = P.sa[ab], sb = P.sb[ab];
    const int np = P.npp[ab];
    double A[3], B[3];
#pragma unroll
    for (int x = 0; x < 3; x++) {
        A[x] = S.xyz[3 * sa + x];
        B[x] = S.xyz[3 * sb + x];
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    double cart[ncart(C::LA) * ncart(C::LB) * ncart(C::LC) * ncart(C::LD)];
    const bool work = threadIdx.x < np * np;
    if (work) pair_block<C>(P, P.pp, ab, A, B, np, threadIdx.x, np * np, blockDim.x, boys, cart);
#pragma unroll
    for (int i = 0; i < na; i++)
#pragma unroll
        for (int j = 0; j < nb; j++) {
            const double v = work ? cart[((i * nb + j) * na + i) * nb + j] : 0.0;
            double s = v;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) s_diag[w][i * nb + j] = s;
        }
    __syncthreads();
    if (w == 0) {
        double m = 0.0;
        if (lane < na * nb) {
            double s = 0.0;
            for (int k = 0; k < nw; k++) s += s_diag[k][lane];
            m = fmax(m, fabs(s));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) Qout[ab] = sqrt(m);
    }
}

template <class C>
static void schwarz_run(const Pairs& P, const Shells& S, const int* list, int n, const double* boys, double* Q,
                        cudaStream_t st)
{
    // one primitive quartet per thread while the blocks' warps fit the chip's
    // 608 schedulers a few times over; with more pairs one warp per pair, whose
    // threads take three each and share one horizontal recursion
    const int threads = n <= 1024 ? SCHWARZ_WIDE : 32;
    if (n > 0) schwarz_kernel<C><<<n, threads, 0, st>>>(P, S, list, n, boys, Q);
}

// Primitive-pair Schwarz factors: for every primitive pair k of shell pair ab
// (one thread per primitive pair, PSW_PAIRS shell pairs per block; one thread
// per shell pair, as before, ran its nine one after another: 17 ms for the
// (dd|dd) pairs of one (H2O)8 bead), qp_k = sqrt(max over functions of
// |(kk|kk)|) with the contraction coefficients included, so that |(ij|kl)| <=
// qp_i qp_l for any primitive quartet (Cauchy-Schwarz for the two charge
// distributions). The pair's primitive data are then reordered by descending
// qp (every field, in place) and qp is stored in that order.
constexpr int PSW_PAIRS = 7;   // shell pairs per block: 63 of 64 threads

template <class C>
__global__ void __launch_bounds__(64) prim_schwarz_kernel(Pairs P, Shells S, const int* __restrict__ list, int n,
                                                          const double* __restrict__ boys, double* pp, float* qp,
                                                          float* qg)
{
    __shared__ float s_q[PSW_PAIRS][PIMD_MAXPP];
    __shared__ int s_perm[PSW_PAIRS][PIMD_MAXPP];
    const int u = threadIdx.x / PIMD_MAXPP, k = threadIdx.x % PIMD_MAXPP;
    const int idx = blockIdx.x * PSW_PAIRS + u;
    const bool mine = u < PSW_PAIRS && idx < n;
    const size_t N = P.n;
    const int ab = mine ? list[idx] : 0;
    const int np = mine ? P.npp[ab] : 0;
    if (k < np) {
        const int sa = P.sa[ab], sb = P.sb[ab];
        double A[3], B[3];
#pragma unroll
        for (int x = 0; x < 3; x++) {
            A[x] = S.xyz[3 * sa + x];
            B[x] = S.xyz[3 * sb + x];
        }
        constexpr int na = nsph(C::LA), nb = nsph(C::LB);
        double cart[ncart(C::LA) * ncart(C::LB) * ncart(C::LC) * ncart(C::LD)];
        pair_block<C>(P, pp, ab, A, B, np, k * np + k, k * np + k + 1, 1, boys, cart);
        double m = 0.0;
        for (int i = 0; i < na; i++)
            for (int j = 0; j < nb; j++) m = fmax(m, fabs(cart[((i * nb + j) * na + i) * nb + j]));
        // rounded up so that the float bound stays an upper bound
        s_q[u][k] = __double2float_ru(sqrt(m) * (1.0 + 1e-6));
    }
    __syncthreads();
    if (mine && k == 0) {
        // insertion sort of the primitive pairs, descending qp (stable)
        int* perm = s_perm[u];
        const float* q = s_q[u];
        for (int a = 0; a < np; a++) {
            int j = a - 1;
            while (j >= 0 && q[perm[j]] < q[a]) {
                perm[j + 1] = perm[j];
                j--;
            }
            perm[j + 1] = a;
        }
    }
    __syncthreads();
    double v[PP_NF];
    if (k < np)
#pragma unroll
        for (int f = 0; f < PP_NF; f++) v[f] = pp[((size_t)f * PIMD_MAXPP + s_perm[u][k]) * N + ab];
    __syncthreads();   // every field is read before any is written
    if (!mine) return;
    float q = 0.0f, g = 0.0f;
    if (k < np) {
#pragma unroll
        for (int f = 0; f < PP_NF; f++) pp[((size_t)f * PIMD_MAXPP + k) * N + ab] = v[f];
        q = s_q[u][s_perm[u][k]];
        g = q * __double2float_ru(2.0 * sqrt(2.0 * fmax(v[PP_EA], v[PP_EB])));
    }
    qp[(size_t)k * N + ab] = q;
    qg[(size_t)k * N + ab] = g;
}

template <class C>
static void prim_schwarz_run(const Pairs& P, const Shells& S, const int* list, int n, const double* boys, double* pp,
                             float* qp, float* qg, cudaStream_t st)
{
    if (n > 0)
        prim_schwarz_kernel<C><<<(n + PSW_PAIRS - 1) / PSW_PAIRS, 64, 0, st>>>(P, S, list, n, boys, pp, qp, qg);
}

}  // namespace pimd
