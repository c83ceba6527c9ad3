// Helpers shared by the FD-subcell kernels and their reverse mode: scratch
// layouts (extended blocks, face fluxes), shell geometry of an element, face
// indexing, and the WENO5-Z interpolation (Sec. III.C.2).
#pragma once
#include "ffe_internal.h"
#include "fp64util.cuh"
#include "physics.cuh"
#include "physics_gen.cuh"
#include "shellmap.cuh"

namespace ffe {

constexpr int NQ = 12;  // reconstructed quantities: 9 evolved + J~ (3)

__device__ __forceinline__ int64_t ext_size(const Dev& d) {
    const int64_t ne = d.nc + 2 * GH;
    return ne * ne * ne;
}
// ext layout: [NQ][chunk][ext_size] indexed by position in the chunk
__device__ __forceinline__ double* ext_at(const Dev& d, int q, int wl) {
    return d.ext + ((int64_t)q * d.chunk + wl) * ext_size(d);
}
__device__ __forceinline__ int64_t nface(const Dev& d) { return (int64_t)(d.nc + 1) * d.nc * d.nc; }
// A face of direction k is m (0..nc) along k, (ta, tb) across; index
// ta + nc tb + nc^2 m, so that the threads of neighbouring lines, which reach
// their faces together, store to neighbouring addresses.
__device__ __forceinline__ int face_index(int nc, int m, int ta, int tb) { return ta + nc * (tb + nc * m); }
// face results: boxes the flux [3][NV][chunk][nface]; flat shells the face states
// [3][NFS][chunk][nface] (k_fd_states); the Kerr-Schild background and the
// adjoint's forward recomputation every physical component j of the flux,
// [3 (k)][3 (j)][NV][chunk][nface]
constexpr int NFS = NQ + NV;
__device__ __forceinline__ double* fstate_at(const Dev& d, int k, int q, int wl) {
    return d.flux + (((int64_t)k * NFS + q) * d.chunk + wl) * nface(d);
}
__device__ __forceinline__ double* flux_at(const Dev& d, int k, int v, int wl) {
    return d.flux + (((int64_t)k * NV + v) * d.chunk + wl) * nface(d);
}
__device__ __forceinline__ double* flux_at_c(const Dev& d, int k, int j, int v, int wl) {
    return d.flux + ((((int64_t)k * 3 + j) * NV + v) * d.chunk + wl) * nface(d);
}
// shell map of element e (its instance's geometry and its index inside the instance)
__device__ __forceinline__ ShellGeo shell_for(const Dev& d, int e, int& el) {
    ShellGeo g;
    g.a = 0.0;   // FD subcells run on shells with x = r v only
    if (d.einst) {
        const InstInfo& in = d.inst[d.einst[e]];
        g.r_in = in.r_in;
        g.c = in.c;
        g.na = in.na;
        g.nr = in.nr;
        el = e - in.e0;
    } else {
        g.r_in = d.shell_rin;
        g.c = d.shell_c;
        g.na = d.shell_na;
        g.nr = d.shell_nr;
        el = e;
    }
    return g;
}

// FD-point geometry of a flat-shell element from the tabulated gnomonic
// coordinates and radii of its rows (Dev::stab): base indices of the element's
// angular and radial rows on the half-cell grid, its wedge axes and side.
struct ShellPts {
    const double *tx, *tw, *tn, *tr, *tir;
    int gx, gy, gr, pn;
    double s, na, nr, c;
};
__device__ __forceinline__ ShellPts shell_pts(const Dev& d, int e, int nc) {
    int el;
    const ShellGeo g = shell_for(d, e, el);
    int ia, ib, ir, w;
    shell_elem(g, el, ia, ib, ir, w);
    ShellPts p;
    const double* t = d.stab + (d.einst ? d.inst[d.einst[e]].tab : 0);
    const int nx = 2 * nc * g.na + 1, nrr = 2 * nc * g.nr + 1;
    p.tx = t;
    p.tw = t + nx;
    p.tn = t + 2 * nx;
    p.tr = t + 3 * nx;
    p.tir = t + 3 * nx + nrr;
    p.gx = 2 * nc * ia;
    p.gy = 2 * nc * ib;
    p.gr = 2 * nc * ir;
    p.pn = (w >> 1) == 0 ? 2 : ((w >> 1) == 1 ? 1 : 0);
    p.s = (w & 1) ? -1.0 : 1.0;
    p.na = g.na;
    p.nr = g.nr;
    p.c = g.c;
    return p;
}
// inverse Jacobian (and the point, if x) at the centre of cell cc
__device__ __forceinline__ void shell_cell(const ShellPts& p, const int* cc, double ij[3][3], double* x) {
    const int hx = p.gx + 2 * cc[0] + 1, hy = p.gy + 2 * cc[1] + 1, hr = p.gr + 2 * cc[2] + 1;
    shell_cell_closed(p.tx[hx], p.tx[hy], p.tw[hx], p.tw[hy], p.tr[hr], p.tir[hr], p.pn, p.s, p.na, p.nr, p.c, ij, x);
}
// unit normal grad xi^k / |grad xi^k| at face m of direction k, tangential cells (ta, tb)
__device__ __forceinline__ void shell_face_normal(const ShellPts& p, int k, int m, int ta, int tb, double* nh) {
    double X, Y;
    if (k == 0) { X = p.tx[p.gx + 2 * m]; Y = 0.0; }
    else if (k == 1) { X = 0.0; Y = p.tx[p.gy + 2 * m]; }
    else { X = p.tx[p.gx + 2 * ta + 1]; Y = p.tx[p.gy + 2 * tb + 1]; }
    shell_normal_closed(k, X, Y, p.pn, p.s, nh);
}

// grad xi^k at the centre of cell cc (row ijk of its inverse Jacobian) times the unit
// normal at face m of direction k next to it: for k = 0 with X_c, T the gnomonic
// coordinates of the centre and the face, na rho/(q (1+X_c^2) r) (1 + X_c T)/sqrt(1 + T^2)
// (likewise k = 1); for k = 2 both are along x^, and it is |grad xi^2|.
__device__ __forceinline__ double shell_grad_normal(const ShellPts& p, int k, const int* cc, int m, const double* ijk) {
    if (k == 2) return p.nr * p.tir[p.gr + 2 * cc[2] + 1] / p.c;
    const int g = k == 0 ? p.gx : p.gy, pt = (p.pn + 1 + k) % 3;
    return ijk[pt] * p.tn[g + 2 * m] * fma(p.tx[g + 2 * cc[k] + 1], p.tx[g + 2 * m], 1.0);
}

__device__ __forceinline__ void axes_of(int dd, int& t1, int& t2) {
    t1 = dd == 0 ? 1 : 0;
    t2 = dd == 2 ? 1 : 2;
}

// number of listed elements in this chunk
__device__ __forceinline__ int chunk_n(const Dev& d, int ci, int w0) {
    const int n = d.counts[ci] - w0;
    return n < 0 ? 0 : (n > d.chunk ? d.chunk : n);
}

// WENO5-Z (point-value interpolation candidates, ideal weights (1, 10, 5)/16,
// Jiang-Shu indicators, Z weights q = 2): the weights
// alpha_k = d_k (1 + t^2/b_k^2), b_k = beta_k + eps, t = b_0 - b_2, are scaled by
// X = b_0^2 b_1^2 b_2^2, so that the normalised combination needs one division:
//   A_k = d_k (X + t^2 prod_{j != k} b_j^2),  value = sum A_k p_k / sum A_k.
// weno5z_combine: the Z-weighted combination of three candidates from their
// indicators b_k (eps included); the ideal weights are taken as (1, 10, 5)
// (scale-free).
// The eps of every WENO5-Z form: weno_eps, zero and values below 2^-1000 as 2^-1000 (the
// reverse mode divides by it; nothing else needs a least value).
__device__ __forceinline__ double indicator_eps(double weno_eps) { return fmax(weno_eps, 9.332636185032189e-302); }

// The weights are homogeneous of degree 0 in the indicators, which are first scaled by
// one power of two, the largest to [1, 2) (exponents only: exact, and products of six
// stay in range), none to less than 2^-250 (a weight that far out is 2^-500).
// Arguments that are not finite stay so.
__device__ __forceinline__ void scale_indicators(double& b0, double& b1, double& b2) {
    const unsigned long long e = umax(fbits(b0), umax(fbits(b1), fbits(b2))) >> 52;   // positive: ordered as integers
    const long long shift = e >= 2047 ? 0 : ((long long)e - 1023) << 52, least = (1023LL - 250) << 52;
    b0 = __longlong_as_double(max(__double_as_longlong(b0) - shift, least));
    b1 = __longlong_as_double(max(__double_as_longlong(b1) - shift, least));
    b2 = __longlong_as_double(max(__double_as_longlong(b2) - shift, least));
}
__device__ __forceinline__ double weno5z_combine(double b0, double b1, double b2, double p0, double p1, double p2) {
    scale_indicators(b0, b1, b2);
    // A_k = d_k (b_k^2 + t^2) P_k with P_k the product of the other two b_j^2
    // is d_k (X + t^2 P_k), X = b_0^2 b_1^2 b_2^2 shared by the three
    const double t = b0 - b2;
    const double t2 = t * t;
    const double q0 = b0 * b0, q1 = b1 * b1, q2 = b2 * b2;
    const double P0 = q1 * q2, P1 = q0 * q2, P2 = q0 * q1;
    const double X = q0 * P0;
    const double A0 = fma(t2, P0, X), A1 = 10.0 * fma(t2, P1, X), A2 = 5.0 * fma(t2, P2, X);
    return fma(A0, p0, fma(A1, p1, A2 * p2)) * recip_nr(A0 + A1 + A2);
}

// Both values at the face between v2 and v3 from the six cells v0..v5 (one face
// at a time: k_fd_flux_faces): uL the
// WENO5-Z value from v0..v4, uR the one from v5..v1 (mirrored).  Everything is
// built from the first differences d_i = v_{i+1} - v_i: the candidates (the
// quadratics through v0..v2, v1..v3, v2..v4 and v3..v5 at the face), the
// second differences a and the one-sided combinations e of the Jiang-Shu
// indicators beta = (13/12) a^2 + (1/4) e^2, of which 4 (beta + eps) enter
// the weights (they are invariant under a common scale of the indicators).
// The two values share two candidates and two second differences.
__device__ __forceinline__ void weno5z_pair(double v0, double v1, double v2, double v3, double v4, double v5,
                                            double eps, double& uL, double& uR) {
    const double d01 = v1 - v0, d12 = v2 - v1, d23 = v3 - v2, d34 = v4 - v3, d45 = v5 - v4;
    const double p123 = fma(0.125, d12, fma(0.375, d23, v2));
    const double p234 = fma(0.625, d23, fma(-0.125, d34, v2));
    const double pL0 = fma(-0.375, d01, fma(0.875, d12, v2));
    const double pR0 = fma(-0.875, d34, fma(0.375, d45, v3));
    const double a012 = d12 - d01, a123 = d23 - d12, a234 = d34 - d23, a345 = d45 - d34;
    const double eL0 = fma(2.0, d12, a012), eL1 = d12 + d23, eL2 = fma(-2.0, d23, a234);
    const double eR0 = fma(-2.0, d34, a345), eR1 = d23 + d34, eR2 = fma(2.0, d23, a123);
    const double c = 13.0 / 3.0, eps4 = 4.0 * indicator_eps(eps);
    const double c123 = c * a123, c234 = c * a234;
    const double bL0 = fma(c * a012, a012, fma(eL0, eL0, eps4));
    const double bL1 = fma(c123, a123, fma(eL1, eL1, eps4));
    const double bL2 = fma(c234, a234, fma(eL2, eL2, eps4));
    const double bR0 = fma(c * a345, a345, fma(eR0, eR0, eps4));
    const double bR1 = fma(c234, a234, fma(eR1, eR1, eps4));
    const double bR2 = fma(c123, a123, fma(eR2, eR2, eps4));
    uL = weno5z_combine(bL0, bL1, bL2, pL0, p123, p234);
    uR = weno5z_combine(bR0, bR1, bR2, pR0, p234, p123);
}

// Reconstruction along one line of cells (one quantity): cell() takes the cell
// two ahead of the current centre c and gives both face values of c -- right:
// the left state of the face to its right, left: the right state of the face to
// its left -- then moves on to c + 1.  A thread that marches a line so does per
// cell what a thread per face does twice: the two values of a cell use the same
// three stencils, hence the same smoothness indicators, and the differences of
// a stencil are those of the next one shifted.  All offsets are taken from the
// centre value.
//
// The smoothness indicators b_k = (13/12) a_k^2 + eps + e_k^2 and the Z weights
// S_k = (1 + T^2/b_k^2) (b_0 b_1 b_2)^2, T = b_0 - b_2, in integers: every term is a
// square, and the weights are sums of two of them, (b_0 b_1 b_2)^2 + (T b_1 b_2)^2 and
// its permutations.  A positive number is m 2^(e - 1022 - 64); products of 64-bit
// fractions m keep the upper half (4 clocks of an SM where an FP64 product takes 16),
// sums the bits that both terms have at the larger one's scale: cut at 2^-57 of the
// larger term, where FP64 rounds each of 16 operations at 2^-53.  Every S_k has a
// scale of its own: a stencil across a jump gets the weight it has (1e-80 and less),
// not one cut at the others' last bit.  No range of indicators overflows; arguments
// that are not finite give finite weights without meaning (the differences they
// multiply are not finite either).
struct Pos {
    unsigned long long m;
    int e;
};
struct ZWeights {
    double s0, s0x5, s1x10, s2, s2x5;   // S_0, 5 S_0, 10 S_1, S_2, 5 S_2
    double right, left;                 // 2 (S_0 + 10 S_1 + 5 S_2) and 2 (5 S_0 + 10 S_1 + S_2)
};
__device__ __forceinline__ Pos pos_of(double x) {
    return {(fbits(x) << 11) | 0x8000000000000000ULL, (int)(fmag(x) >> 52)};
}
__device__ __forceinline__ Pos pos_square(double x) {   // 2^62 <= m; a zero counts as 2^-2044
    const Pos p = pos_of(x);
    return {__umul64hi(p.m, p.m), 2 * p.e - 1022};
}
__device__ __forceinline__ Pos pos_add(Pos x, Pos y) {
    const int e = max(x.e, y.e) + 1;
    return {(x.m >> min(e - x.e, 63)) + (y.m >> min(e - y.e, 63)), e};
}
// m >= 2^32 to 2^63 <= m
__device__ __forceinline__ Pos pos_norm(Pos x) {
    const int lz = __clz((int)(x.m >> 32));
    return {x.m << lz, x.e - lz};
}
// m 2^e rounded to nearest, for 2^63 <= m and for any positive m
__device__ __forceinline__ double norm_double(unsigned long long m, int e) {
    return __longlong_as_double((long long)((m >> 11) + ((m >> 10) & 1ULL) + ((unsigned long long)(1085 + e) << 52)));
}
__device__ __forceinline__ double pos_double(unsigned long long m, int e) {
    const int lz = __clzll((long long)m);
    return norm_double(m << lz, e - lz);
}
// b_k of magnitude 2^63 <= m
__device__ __forceinline__ ZWeights z_weights(Pos b0, Pos b1, Pos b2) {
    const int eM = max(b0.e, b2.e);
    const unsigned long long u = b0.m >> min(eM - b0.e, 63), v = b2.m >> min(eM - b2.e, 63), tt = u > v ? u - v : v - u;
    // T = 0: its terms lie below all others, else they would shift the first square away
    const int lzt = __clzll((long long)(tt | 1ULL)), et = tt ? eM - lzt : -(1 << 20);
    const unsigned long long ft = tt << lzt;
    // half the right shifts of T's terms against the first square, none of them below the least
    const int s0 = b0.e - et, s1 = b1.e - et, s2 = b2.e - et, least = min(0, min(s0, min(s1, s2)));
    const int n0 = 2 * (s0 - least), n1 = 2 * (s1 - least), n2 = 2 * (s2 - least), nX = -2 * least;
    const unsigned long long c0 = __umul64hi(b1.m, b2.m), c1 = __umul64hi(b0.m, b2.m), c2 = __umul64hi(b0.m, b1.m);
    const unsigned long long r0 = __umul64hi(ft, c0), r1 = __umul64hi(ft, c1), r2 = __umul64hi(ft, c2);
    const unsigned long long Y = __umul64hi(b1.m, c1);
    const unsigned long long q0 = __umul64hi(r0, r0), q1 = __umul64hi(r1, r1), q2 = __umul64hi(r2, r2), qX = __umul64hi(Y, Y);
    // a weight at its larger term's scale, to 2^63 <= m (the terms are 2^58 or more there; T = 0 leaves X alone)
    auto sum = [&](unsigned long long q, int n) -> Pos {
        const int k = min(n, nX);
        const unsigned long long m = (qX >> min(nX - k + 1, 63)) + (q >> min(n - k + 1, 63));
        const int lz = __clz((int)(m >> 32));
        return {m << lz, 1 - lz - min(k, 1000)};
    };
    const Pos S0 = sum(q0, n0), S1 = sum(q1, n1), S2 = sum(q2, n2);
    // the sums at the largest term's scale (2^58 or more there); five bits of room
    auto top = [](unsigned long long q, int n) { return (unsigned)(q >> 32) >> min(n, 31); };
    const int room = 5 - min(5, __clz((int)(top(q0, n0) | top(q1, n1) | top(q2, n2) | top(qX, nX))));
    auto down = [&](unsigned long long q, int n) { return q >> min(n + room, 63); };
    const unsigned long long X = 16 * down(qX, nX), t0 = down(q0, n0), t1 = X + 10 * down(q1, n1), t2 = down(q2, n2);
    ZWeights w;
    w.s0 = norm_double(S0.m, S0.e);
    w.s0x5 = pos_double(5 * (S0.m >> 3), S0.e + 3);
    w.s1x10 = pos_double(5 * (S1.m >> 3), S1.e + 4);
    w.s2 = norm_double(S2.m, S2.e);
    w.s2x5 = pos_double(5 * (S2.m >> 3), S2.e + 3);
    w.right = pos_double(t0 + t1 + 5 * t2, room + 1);
    w.left = pos_double(5 * t0 + t1 + t2, room + 1);
    return w;
}

// WENO5-Z: with a_k the second difference of stencil k (left, centred, right) and
// e_k its slope at the centre, the candidate at the face +-1/2 is
// v_c + a_k / 8 +- e_k / 2, and beta_k = (13/12) a_k^2 + e_k^2 (the kept per-stencil
// values are a and k = (13/12) a^2 + eps); ideal weights (1, 10, 5) towards the
// right face and (5, 10, 1) towards the left one.  Twice the candidates' offsets from
// v_c are one operation each from the differences.  25 FP64 operations per cell and
// quantity, the pipe that bounds these kernels (87 in a thread per face).  Every
// offset is formed from its own stencil's differences: beside a jump, the values of the
// smooth side are as accurate as its cells (candidates by their differences from the
// central one, 23 operations, and weights at one scale leave 2^-54 of the jump there;
// two steps of the 64x8x8 current sheet 9.46 -> 9.60 ms, 19 blocks 88 -> 91 us).
struct Weno5zLine {
    double dA, dB, aA, aB, vc, vn;
    Pos kA, kB, eps;
    __device__ __forceinline__ Pos curv(double a) const {
        const Pos q = pos_square(a);
        return pos_add({__umul64hi(q.m, 0x8aaaaaaaaaaaaaabULL), q.e + 1}, eps);   // 13/24 2^64
    }
    __device__ __forceinline__ void init(double v0, double v1, double v2, double v3, double weno_eps) {
        eps = pos_of(indicator_eps(weno_eps));
        const double d01 = v1 - v0;
        dA = v2 - v1;
        dB = v3 - v2;
        aA = dA - d01;
        aB = dB - dA;
        kA = curv(aA);
        kB = curv(aB);
        vc = v2;
        vn = v3;
    }
    template <bool LEFT, bool RIGHT>
    __device__ __forceinline__ void cell(double v4, double& left, double& right) {
        const double dC = v4 - vn, aC = dC - dB;
        const Pos kC = curv(aC);
        const double e0 = fma(0.5, aA, dA), e1 = fma(0.5, aB, dA), e2 = fma(-0.5, aC, dB);   // slopes at the centre
        const ZWeights S = z_weights(pos_norm(pos_add(pos_square(e0), kA)), pos_norm(pos_add(pos_square(e1), kB)),
                                     pos_norm(pos_add(pos_square(e2), kC)));
        if (RIGHT)
            right = fma(fma(S.s0, fma(0.75, aA, dA), fma(S.s1x10, fma(0.75, aB, dA), S.s2x5 * fma(-0.25, aC, dB))),
                        recip_nr3(S.right), vc);
        if (LEFT)
            left = fma(fma(-S.s0x5, fma(0.25, aA, dA), fma(-S.s1x10, fma(0.25, aB, dA), -S.s2 * fma(-0.75, aC, dB))),
                       recip_nr3(S.left), vc);
        dA = dB; dB = dC;
        aA = aB; aB = aC;
        kA = kB; kB = kC;
        vc = vn; vn = v4;
    }
};

// MP5 (Suresh & Huynh, J. Comput. Phys. 136, 83 (1997)) on the 5-point
// interpolant (3, -20, 90, 60, -5)/128, alpha = 4: the interpolant where its
// offset d from v_c lies between 0 and v_MP - v_c = minmod(v_+ - v_c, 4 (v_c -
// v_-)), else its median with the bounds built from v_UL, v_MD, v_LC and the
// minmod4 curvatures.  Both bounds contain the centre (lower <= v_c <= upper), so
// the median is d limited to [-N, P].  Only magnitudes and signs are compared, as
// integers: an FP64 comparison takes the FP64 pipe, 1/32 of the integer rate.
__device__ __forceinline__ double minmod4(double a, double b, double c, double d) {
    const bool s = fneg(a);
    if (fneg(b) != s || fneg(c) != s || fneg(d) != s) return 0.0;
    const unsigned long long m = umin(umin(fmag(a), fmag(b)), umin(fmag(c), fmag(d)));
    return __longlong_as_double((long long)(s ? m | 0x8000000000000000ULL : m));
}

// d limited to the median bounds of one face: dn the difference towards the
// face's far cell, du4 four times the upwind one, md and lc the offsets of v_MD
// and v_LC.  NaN stays NaN.
__device__ __forceinline__ double mp5_limit(double d, double dn, double du4, double md, double lc) {
    auto part = [](double x, bool neg) { return fneg(x) == neg ? fmag(x) : 0ULL; };
    const bool neg = fneg(d);
    const unsigned long long lim = umin(umax(part(dn, neg), part(md, neg)), umax(part(du4, neg), part(lc, neg)));
    const unsigned long long m = fmag(d);
    if (m <= lim || m > 0x7ff0000000000000ULL) return d;
    return __longlong_as_double((long long)(neg ? lim | 0x8000000000000000ULL : lim));
}

struct Mp5Line {
    double d0, dA, dB, aA, aB, vc, vn;
    __device__ __forceinline__ void init(double v0, double v1, double v2, double v3, double) {
        d0 = v1 - v0;
        dA = v2 - v1;
        dB = v3 - v2;
        aA = dA - d0;
        aB = dB - dA;
        vc = v2;
        vn = v3;
    }
    // the interpolant's offset is inside [0, minmod(dn, du4)]
    static __device__ __forceinline__ bool inside(double d, double dn, double du4) {
        const unsigned long long m = fmag(d);
        return m == 0 || (fneg(d) == fneg(dn) && fneg(d) == fneg(du4) && m <= umin(fmag(dn), fmag(du4)));
    }
    template <bool LEFT, bool RIGHT>
    __device__ __forceinline__ void cell(double v4, double& left, double& right) {
        const double dC = v4 - vn, aC = dC - dB;
        // (-3 d0 + 17 dA + 55 dB - 5 dC)/128 and its mirror image
        double r = fma(-0.0234375, d0, fma(0.1328125, dA, fma(0.4296875, dB, -0.0390625 * dC)));
        double l = fma(0.0234375, dC, fma(-0.1328125, dB, fma(-0.4296875, dA, 0.0390625 * d0)));
        const double dA4 = 4.0 * dA, dB4 = -4.0 * dB;
        const bool okr = !RIGHT || inside(r, dB, dA4), okl = !LEFT || inside(l, -dA, dB4);
        if (!(okr && okl)) {
            const double mp = minmod4(fma(4.0, aB, -aC), fma(4.0, aC, -aB), aB, aC);   // curvature at the right face
            const double mm = minmod4(fma(4.0, aB, -aA), fma(4.0, aA, -aB), aB, aA);   // at the left face
            if (!okr) r = mp5_limit(r, dB, dA4, 0.5 * (dB - mp), fma(4.0 / 3.0, mm, 0.5 * dA));
            if (!okl) l = mp5_limit(l, -dA, dB4, -0.5 * (dA + mm), fma(4.0 / 3.0, mp, -0.5 * dB));
        }
        if (RIGHT) right = vc + r;
        if (LEFT) left = vc + l;
        d0 = dA; dA = dB; dB = dC;
        aA = aB; aB = aC;
        vc = vn; vn = v4;
    }
};

template <int RECON> struct LineOf { using type = Weno5zLine; };
template <> struct LineOf<FFE_RECON_MP5> { using type = Mp5Line; };

// Where line (ta, tb) of direction k starts in an extended block: its first ghost,
// and the step along it.
__device__ __forceinline__ int64_t line_start(int k, int ta, int tb, int nc, int64_t& stride) {
    const int64_t ne = nc + 2 * GH;
    int t1, t2;
    axes_of(k, t1, t2);
    const int64_t st[3] = {1, ne, ne * ne};
    stride = st[k];
    return (ta + GH) * st[t1] + (tb + GH) * st[t2];
}

// Reconstructs two quantities along one line of nc cells with 3 ghosts at each
// end (pa, pb: the line's first ghost; sb: sign bit flipped in every value of
// the second) and calls emit(m, La, Ra, Sa, Lb, Rb, Sb) at its faces m = 0..nc in
// order: left and right states and the sum of the two cells at the face.  Two
// quantities give a thread two independent chains of operations.
template <class Line, class Emit>
__device__ __forceinline__ void recon_lines(const double* pa, const double* pb, int64_t stride, unsigned long long sb,
                                            int nc, double eps, Emit emit) {
    auto b_at = [&](const double* p) { return __longlong_as_double((long long)(fbits(*p) ^ sb)); };
    Line A, B;
    A.init(pa[0], pa[stride], pa[2 * stride], pa[3 * stride], eps);
    B.init(b_at(pb), b_at(pb + stride), b_at(pb + 2 * stride), b_at(pb + 3 * stride), eps);
    pa += 4 * stride;
    pb += 4 * stride;
    double La, Lb, Ra, Rb, ca = A.vc, cb = B.vc;
    A.template cell<false, true>(*pa, Ra, La);
    B.template cell<false, true>(b_at(pb), Rb, Lb);
#pragma unroll 1
    for (int m = 0; m < nc; ++m) {
        pa += stride;
        pb += stride;
        double na, nb;
        const double Sa = ca + A.vc, Sb = cb + B.vc;
        ca = A.vc;
        cb = B.vc;
        A.template cell<true, true>(*pa, Ra, na);
        B.template cell<true, true>(b_at(pb), Rb, nb);
        emit(m, La, Ra, Sa, Lb, Rb, Sb);
        La = na;
        Lb = nb;
    }
    const double Sa = ca + A.vc, Sb = cb + B.vc;
    A.template cell<true, false>(pa[stride], Ra, La);
    B.template cell<true, false>(b_at(pb + stride), Rb, Lb);
    emit(nc, La, Ra, Sa, Lb, Rb, Sb);
}

// The flat flux along direction k couples the reconstructed quantities in five
// pairs (a, b) with a sign s: F_a = s b, F_b = s a -- (E_k, psi), (B_k, phi),
// (E_i, B_j) with s = 1, (E_j, B_i) with s = -1 for (k, i, j) cyclic -- and
// (q, J_k) with F_q = J_k only; the other two components of J~ do not enter.
__device__ __forceinline__ void flux_pair(int k, int pr, int& a, int& b, bool& neg) {
    const int i = k == 2 ? 0 : k + 1, j = k == 0 ? 2 : k - 1;
    neg = pr == 3;
    a = pr == 0 ? k : (pr == 1 ? 3 + k : (pr == 2 ? i : (pr == 3 ? j : 8)));
    b = pr == 0 ? 6 : (pr == 1 ? 7 : (pr == 2 ? 3 + j : (pr == 3 ? 3 + i : NV + k)));
}
constexpr int FLUX_PAIRS = 5;

// Rusanov flux (lambda = 1) of a pair from its states, b carrying the sign s:
// F_a = (b_L + b_R)/2 - (a_R - a_L)/2 and F_b likewise, with the corrector
// F - (F_m - 2 F + F_p)/6 = (4/3) F - (F_m + F_p)/6 (S: the sum of the two cells).
__device__ __forceinline__ void rusanov_pair(double La, double Ra, double Sa, double Lb, double Rb, double Sb, bool corr,
                                             double& Fa, double& Fb) {
    const double p = La + Lb, m = Rb - Ra;
    if (corr) {
        Fa = fma(-1.0 / 6.0, Sb, (2.0 / 3.0) * (p + m));
        Fb = fma(-1.0 / 6.0, Sa, (2.0 / 3.0) * (p - m));
    } else {
        Fa = 0.5 * (p + m);
        Fb = 0.5 * (p - m);
    }
}

// Reverse mode of the two face values of a cell (Weno5zLine, WENO5-Z): from the
// adjoints yl, yr of its left and right value, the adjoints of the window's
// differences and scaled second differences (h = a/8), added to them:
// hb0..hb2 (of h at c-1, c, c+1), dAb, dBb (of the differences left and right
// of c); the centre value's adjoint is yl + yr.  With S_k = (b_k^2 + t^2) P_k,
// t = b_0 - b_2, P_k the product of the other two b_j^2, and W_k = dL/dS_k summed
// over both values (y d_k (g_k - value) / sum A):
//   dL/db_0 = 2 (t T + b_0 (W_0 P_0 + W_1 s_1 b_2^2 + W_2 s_2 b_1^2)),
//   dL/db_1 = 2 b_1 (W_0 s_0 b_2^2 + W_1 P_1 + W_2 s_2 b_0^2),
//   dL/db_2 = 2 (-t T + b_2 (W_0 s_0 b_1^2 + W_1 s_1 b_0^2 + W_2 P_2)),
// T = sum_k W_k P_k, s_k = b_k^2 + t^2.  The weights are homogeneous of degree 0 in
// the b_k, so these are first scaled exactly by the power of two of their maximum;
// the S_k are then O(1) and their derivatives stay in range.
struct Weno5zLineVjp {
    double dA, dB, hA, hB, kA, kB, vn, eps;
    __device__ __forceinline__ double curv(double h) const { return fma((13.0 / 12.0 * 64.0) * h, h, eps); }
    __device__ __forceinline__ void init(double v0, double v1, double v2, double v3, double weno_eps) {
        eps = indicator_eps(weno_eps);
        const double d01 = v1 - v0;
        dA = v2 - v1;
        dB = v3 - v2;
        hA = 0.125 * (dA - d01);
        hB = 0.125 * (dB - dA);
        kA = curv(hA);
        kB = curv(hB);
        vn = v3;
    }
    __device__ __forceinline__ void cell(double v4, double yl, double yr, double& hb0, double& hb1, double& hb2, double& dAb,
                                         double& dBb) {
        const double dC = v4 - vn, hC = 0.125 * (dC - dB), kC = curv(hC);
        const double e0 = fma(4.0, hA, dA), e1 = fma(4.0, hB, dA), e2 = fma(-4.0, hC, dB);
        const double c0 = fma(e0, e0, kA), c1 = fma(e1, e1, kB), c2 = fma(e2, e2, kC);
        // positive: ordered as integers
        const double sc = pow2_inv_scale(__longlong_as_double((long long)umax(fbits(c0), umax(fbits(c1), fbits(c2)))));
        double b0 = c0, b1 = c1, b2 = c2;
        scale_indicators(b0, b1, b2);
        const double t = b0 - b2, t2 = t * t;
        const double q0 = b0 * b0, q1 = b1 * b1, q2 = b2 * b2;
        const double s0 = q0 + t2, s1 = q1 + t2, s2 = q2 + t2;
        const double P0 = q1 * q2, P1 = q0 * q2, P2 = q0 * q1;
        const double S0 = s0 * P0, S1 = 10.0 * (s1 * P1), S2 = s2 * P2;
        // The candidates differ from the central one by u = h_1 - h_0 and w = h_2 - h_1 only:
        // right (weights 1, 10, 5) -3 u and -w, left (5, 10, 1) u and 3 w; vr, vl: the values
        // less the central candidate
        const double T2 = 5.0 * S2, T0 = 5.0 * S0;
        const double iR = recip_nr((S0 + S1) + T2), iL = recip_nr((T0 + S1) + S2);
        const double u = hB - hA, w = hC - hB, x0 = S0 * u, x2 = S2 * w;
        const double vr = fma(-3.0, x0, -5.0 * x2) * iR, vl = fma(5.0, x0, 3.0 * x2) * iL;
        const double y = yr * iR, z = yl * iL;
        const double ub = S0 * fma(5.0, z, -3.0 * y), wb = S2 * fma(3.0, z, -5.0 * y);   // of u and w
        const double y5 = 5.0 * y, z5 = 5.0 * z;
        const double W0 = fma(y, fma(-3.0, u, -vr), z5 * (u - vl));
        const double W1 = -2.0 * fma(y5, vr, z5 * vl);
        const double W2 = fma(-y5, w + vr, z * fma(3.0, w, -vl));
        const double W0P0 = W0 * P0, W0s0 = W0 * s0, W1s1 = W1 * s1, W2s2 = W2 * s2;
        const double T = fma(W1, P1, fma(W2, P2, W0P0));
        const double X0 = fma(W1s1, q2, fma(W2s2, q1, W0P0));
        const double X1 = fma(W0s0, q2, fma(W2s2, q0, W1 * P1));
        const double X2 = fma(W0s0, q1, fma(W1s1, q0, W2 * P2));
        const double sc4 = 4.0 * sc;   // B_k: twice the adjoint of b_k
        const double B0 = sc4 * fma(t, T, b0 * X0), B1 = sc4 * (b1 * X1), B2 = sc4 * fma(-t, T, b2 * X2);
        // b = e^2 + K h^2 + eps: to e (slopes) and h
        const double E0 = e0 * B0, E1 = fma(e1, B1, 0.5 * (yr - yl)), E2 = e2 * B2;
        constexpr double K = 13.0 / 12.0 * 64.0;
        hb0 += fma(K * hA, B0, fma(4.0, E0, -ub));
        hb1 += fma(K * hB, B1, fma(4.0, E1, (yr + yl) + (ub - wb)));
        hb2 += fma(K * hC, B2, fma(-4.0, E2, wb));
        dAb += E0 + E1;
        dBb += E2;
        dA = dB; dB = dC;
        hA = hB; hB = hC;
        kA = kB; kB = kC;
        vn = v4;
    }
};

// J~ (drift, full) at cell c of FD element e
__device__ __forceinline__ void current_fd_cell(const Dev& d, int e, int c, const Field& U, const Field& J) {
    if (d.mask[e] != 1 || c >= esz(d, e).ncell) return;
    const int64_t p = fdb(d, e) + c;
    double u[NV], jd[3], jf[3];
    for (int v = 0; v < NV; ++v) u[v] = U.fd(v)[p];
    if (d.ks) {
        PM m;
        load_pm(d.metfd, (int64_t)d.E * d.ncell, (int64_t)e * d.ncell + c, m);
        current_gen(u, m, d.eta, jd, jf);
    } else {
        current_flat(u, d.eta, jd, jf);
    }
    for (int k = 0; k < 3; ++k) { J.fd(k)[p] = jd[k]; J.fd(3 + k)[p] = jf[k]; }
}

// face fi of direction k: position m along k, tangential (ta, tb); false past the element's faces
__device__ __forceinline__ bool face_coords(int64_t fi, int nc, int& m, int& ta, int& tb) {
    const int64_t nf = (int64_t)(nc + 1) * nc * nc;
    if (fi >= nf) return false;
    m = (int)(fi % (nc + 1));
    ta = (int)((fi / (nc + 1)) % nc);
    tb = (int)(fi / ((int64_t)(nc + 1) * nc));
    return true;
}

}  // namespace ffe
