// DG-side kernels of libffe (flat metric, affine box elements).
//
// k_dg_substep fuses, per DG element (one CTA, one thread per LGL node):
//   volume term  -(d xi^k/d x^j) D_k F^j  (Sec. III.A, nodal DG-SEM),
//   the Rusanov boundary correction lifted with the lumped LGL mass (Sec. III.C.2 flux),
//   the explicit sources, the explicit part of the IMEX-SSP3(4,3,3) stage, the
//   exponential filter (Sec. III.A) of that explicit update, the pointwise stiff
//   solve (Sec. III.B), the optional algebraic clamp (Sec. II.B) and the
//   troubled-cell indicator (Sec. III.C.3).  Filtering before the solve keeps
//   every state the explicit right-hand side sees a solve output: a filter after
//   the solve re-creates a parallel E~ that the eta-current of the q~ flux
//   amplifies by eta (unstable for eta dt >> 1).
#include <cstdio>

#include "dgfilter.cuh"
#include "dgtci.cuh"
#include "fd_common.cuh"
#include "ffe_internal.h"
#include "physics.cuh"
#include "physics_gen.cuh"
#include "stage.cuh"

namespace ffe {

thread_local int64_t g_launch_counter = 0;

template <int P>
struct DGK {
    static constexpr int np1 = P + 1;
    static constexpr int nn = np1 * np1 * np1;
    static constexpr int nf = np1 * np1;
    static constexpr int NT = ((nn + 31) / 32) * 32;
    static constexpr int FR = (6 * nf + NT - 1) / NT;   // face nodes per thread
    // CTAs per SM the registers are bounded for
    static constexpr int CTAS = P == 6 ? 2 : 4;
    // shared doubles: U[9][nn] (later the filter's buffer) | dU/dt[9][nn] |
    // fixed point: U and J [12][nn] (later the filter's and the indicator's fields) | red[2] | D scaled by the
    // element's d xi/d x, per axis [3][np1][np1]
    static constexpr int SMEM = (30 * nn + 2 + 3 * nf) * 8;
};

// ---------------------------------------------------------------------------
// Work lists of the mask: FD elements and, per order, DG elements.
__device__ __forceinline__ int list_of(const Dev& d, int e, int** list) {
    if (d.mask[e] != 0) { *list = d.fd_list; return 1; }
    if (!d.dg_list_lo || elem_P(d, e) == d.P) { *list = d.dg_list; return 0; }
    if (elem_P(d, e) == d.P - 1) { *list = d.dg_list_lo; return 6; }
    *list = d.dg_list_lo2;
    return 7;
}

__global__ void k_build_lists(Dev d) {
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= d.E) return;
    int* list;
    const int c = list_of(d, e, &list);
    list[atomicAdd(&d.counts[c], 1)] = e;
}

// The same in one CTA, which clears the counters itself.
__global__ void __launch_bounds__(1024) k_build_lists_small(Dev d, int clear) {
    __shared__ int n[8];
    if (threadIdx.x < 8) n[threadIdx.x] = 0;
    __syncthreads();
    for (int e = threadIdx.x; e < d.E; e += blockDim.x) {
        int* list;
        const int c = list_of(d, e, &list);
        list[atomicAdd(&n[c], 1)] = e;
        if (clear & LISTS_STEP) d.switched[e] = 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        d.counts[0] = n[0];
        d.counts[1] = n[1];
        if (d.dg_list_lo) {
            d.counts[6] = n[6];
            d.counts[7] = n[7];
        }
        if (clear & (LISTS_FLAGS | LISTS_STEP)) d.counts[2] = 0;
        if (clear & LISTS_STEP) d.counts[3] = 0;
    }
}

// One CTA up to 8192 elements: 8 loads in a row per thread cost less than the two
// to five clears that the grid version needs before it (each a node of its own in
// a step's graph).
void launch_build_lists(const Dev& d, cudaStream_t st, int clear) {
    const bool small = d.E <= 8192;
    if (!small) {
        cudaMemsetAsync(d.counts, 0, 2 * sizeof(int), st);
        if (d.dg_list_lo) cudaMemsetAsync(d.counts + 6, 0, 2 * sizeof(int), st);
        if (clear & LISTS_STEP) {
            cudaMemsetAsync(d.counts + 2, 0, 2 * sizeof(int), st);
            cudaMemsetAsync(d.switched, 0, d.E, st);
        } else if (clear & LISTS_FLAGS) {
            cudaMemsetAsync(d.counts + 2, 0, sizeof(int), st);
        }
    }
    prof_begin("build_lists", st);
    if (small) k_build_lists_small<<<1, 1024, 0, st>>>(d, clear);
    else k_build_lists<<<(d.E + 255) / 256, 256, 0, st>>>(d);
    prof_end(st);
    g_launch_counter += 1;
}

// ---------------------------------------------------------------------------
// J~ (drift, full) at every DG node of DG elements and at the cells of the FD
// list (counts[1], as built by k_build_lists).
__global__ void k_current(Dev d, Field U, Field J) {
    int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p = tid; p < d.ndg; p += stride) {
        const int e = (int)(p / d.nn);
        if (d.mask[e] != 0 || (int)(p % d.nn) >= esz(d, e).nn) continue;
        double u[NV], jd[3], jf[3];
        for (int v = 0; v < NV; ++v) u[v] = U.dg(v)[p];
        if (d.ks) {
            PM m;
            load_pm(d.met, d.ndg, p, m);
            current_gen(u, m, d.eta, jd, jf);
        } else {
            current_flat(u, d.eta, jd, jf);
        }
        for (int c = 0; c < 3; ++c) { J.dg(c)[p] = jd[c]; J.dg(3 + c)[p] = jf[c]; }
    }
    const int64_t n = (int64_t)d.counts[1] * d.ncell;
    for (int64_t q = tid; q < n; q += stride) current_fd_cell(d, d.fd_list[q / d.ncell], (int)(q % d.ncell), U, J);
}

void launch_current(const Dev& d, Field U, Field J, cudaStream_t st) {
    prof_begin("current", st);
    k_current<<<d.nsm * 8, 256, 0, st>>>(d, U, J);
    prof_end(st);
    g_launch_counter += 1;
}

// ---------------------------------------------------------------------------
// Stages 1 and 2 are pointwise: U1 = solve(u_n), G1 = G(U1); U2 = solve(u_n - dt a G1), G2 = G(U2);
// J~(U2), which the first right-hand side reads, comes with the second solve.
// Over the DG nodes of DG elements and the cells of the FD list (built first).
__device__ __forceinline__ void stage12_point(const Dev& d, const SolveK& k, bool isfd, int64_t p, const Field& un,
                                              const Field& Ua, const Field& G1, const Field& G2, const Field& J) {
    auto at = [&](const Field& f, int v) { return (isfd ? f.fd(v) : f.dg(v)) + p; };
    double u[NV], U1[NV], jp[3], ib2, g1[NG], g2[NG], jd[3], jf[3];
    for (int v = 0; v < NV; ++v) U1[v] = u[v] = *at(un, v);
    bool ok = implicit_stage_flat(U1, d, k, jp, ib2);
    stage_G_flat(U1, d, jp, g1);
    u[0] = fma(-k.dta, g1[0], u[0]);
    u[1] = fma(-k.dta, g1[1], u[1]);
    u[2] = fma(-k.dta, g1[2], u[2]);
    u[6] = fma(-k.dta, g1[3], u[6]);
    u[7] = fma(-k.dta, g1[4], u[7]);
    ok &= implicit_stage_flat(u, d, k, jp, ib2);
    if (!ok) atomic_status(d, 2);
    stage_G_flat(u, d, jp, g2);
    stage_current_flat(u, jp, ib2, jd, jf);
    for (int v = 0; v < NV; ++v) *at(Ua, v) = u[v];
    for (int c = 0; c < NG; ++c) { *at(G1, c) = g1[c]; *at(G2, c) = g2[c]; }
    for (int c = 0; c < 3; ++c) { *at(J, c) = jd[c]; *at(J, 3 + c) = jf[c]; }
}

__global__ void k_stage12(Dev d, Field un, Field Ua, Field G1, Field G2, Field J) {
    int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p = tid; p < d.ndg; p += stride) {
        const int e = (int)(p / d.nn);
        if (d.mask[e] != 0 || (int)(p % d.nn) >= esz(d, e).nn) continue;
        stage12_point(d, solve_k(d, e), false, p, un, Ua, G1, G2, J);
    }
    // FD cells: the elements of the FD list only (an FD slot pool may be mostly empty)
    const int64_t nfdq = (int64_t)d.counts[1] * d.ncell;
    for (int64_t q = tid; q < nfdq; q += stride) {
        const int e = d.fd_list[q / d.ncell];
        const int c = (int)(q % d.ncell);
        if (c >= esz(d, e).ncell) continue;
        stage12_point(d, solve_k(d, e), true, fdb(d, e) + c, un, Ua, G1, G2, J);
    }
}

void launch_stage12(const Dev& d, Field un, Field Ua, Field G1, Field G2, Field J, cudaStream_t st) {
    prof_begin("stage12", st);
    k_stage12<<<d.nsm * 8, 256, 0, st>>>(d, un, Ua, G1, G2, J);
    prof_end(st);
    g_launch_counter += 1;
}

// tangential node coordinates of face direction dd: t1 < t2 are the other two axes
__device__ __forceinline__ void face_axes(int dd, int& t1, int& t2) {
    t1 = dd == 0 ? 1 : 0;
    t2 = dd == 2 ? 1 : 2;
}

template <int P>
__device__ __forceinline__ int node_index(int c0, int c1, int c2) {
    constexpr int np1 = P + 1;
    return c0 + np1 * (c1 + np1 * c2);
}

// External state at face node (face f, tangential a, b) of element e for the DG lift.
template <int P>
__device__ void dg_external_state(const Dev& d, const SubArgs& a, int e, int f, int ta, int tb,
                                  const double* Ui, const double* xnode, double* Ue, double* Je) {
    constexpr int np1 = P + 1;
    constexpr int nn = np1 * np1 * np1;
    const Tables& T = *d.tab;
    int dd = f >> 1, s = f & 1;
    int t1, t2;
    face_axes(dd, t1, t2);
    int nb = d.nbr[e * 6 + f];
    double jd[3];
    if (nb >= 0) {
        int f2 = d.nbr_face[e * 6 + f];
        int c[3];
        c[f2 >> 1] = (f2 & 1) ? P : 0;
        c[t1] = ta;
        c[t2] = tb;
        if (d.mask[nb] == 0) {
            int64_t p = (int64_t)nb * nn + node_index<P>(c[0], c[1], c[2]);
            for (int v = 0; v < NV; ++v) Ue[v] = a.Uin.dg(v)[p];
            for (int q = 0; q < 3; ++q) Je[q] = a.J.dg(3 + q)[p];
            return;
        }
        // FD neighbour: its FD->DG projection evaluated at this node (6-point
        // stencils), for the state and for its current J~ (the current of the
        // projected state would carry the projection error of E~.B~ times eta),
        // from the face traces face_trace left for it (same face axes: boxes)
        (void)T;
        const int nfm = d.np1 * d.np1;
        const double* tr = d.ftr + ((int64_t)fd_slot_of(d, nb) * 6 + f2) * 12 * nfm + ta + np1 * tb;
        for (int v = 0; v < NV; ++v) Ue[v] = tr[v * nfm];
        for (int q = 0; q < 3; ++q) Je[q] = tr[(NV + q) * nfm];
        return;
    }
    int kind = d.bc[e * 6 + f];
    if (kind == FFE_BC_DIRICHLET) {
        int bfs = d.bface[e * 6 + f];
        const double* src = d.bdg + (int64_t)bfs * NV * np1 * np1;
        for (int v = 0; v < NV; ++v) Ue[v] = src[v * np1 * np1 + ta + np1 * tb];
    } else if (kind == FFE_BC_NO_INCOMING) {
        double n[3] = {0.0, 0.0, 0.0};
        n[dd] = s ? 1.0 : -1.0;
        bc_no_incoming_flat(Ui, n, Ue);
    } else if (kind == FFE_BC_OUTFLOW) {
        for (int v = 0; v < NV; ++v) Ue[v] = Ui[v];
    } else {
        bc_star_flat(Ui, xnode, d.omega, Ue);
    }
    current_flat(Ue, d.eta, jd, Je);
}

// The volume term of equation q (as numbered in U) takes D_k of variable term_var(q, k)
// (9..11: J~) along axis k, with the sign term_neg(q, k).
__host__ __device__ constexpr int term_var(int q, int k) {
    return q < 3 ? (q == k ? 6 : 6 - q - k) : (q < 6 ? (q - 3 == k ? 7 : 6 - q - k) : (q == 6 ? k : (q == 7 ? 3 + k : 9 + k)));
}
__host__ __device__ constexpr bool term_neg(int q, int k) {
    return q >= 6 || q % 3 == k || (q < 3) == ((q + 3 - k) % 3 == 1);
}

// The volume term in FP64, for elements whose values fixed point does not hold.
template <int P>
__device__ __forceinline__ void volume_fp64(Field J, int64_t eb, const double* sU, const double* sD, double* r) {
    constexpr int np1 = P + 1, nf = np1 * np1, nn = nf * np1;
    const int tid = threadIdx.x, i = tid % np1, j = (tid / np1) % np1, k = tid / nf;
    const double *Dx = sD + np1 * i, *Dy = sD + nf + np1 * j, *Dz = sD + 2 * nf + np1 * k;
    const int ox = np1 * (j + np1 * k), oy = i + nf * k, oz = i + np1 * j;
    auto U = [&](int v, int idx) { return sU[v * nn + idx]; };
    double eX = -J.dg(0)[eb + tid], eY = -J.dg(1)[eb + tid], eZ = -J.dg(2)[eb + tid];
    double bX = 0.0, bY = 0.0, bZ = 0.0, ps = U(8, tid), ph = 0.0, qq = 0.0;
#pragma unroll 1
    for (int m = 0; m < np1; ++m) {
        const int ix = ox + m, iy = oy + np1 * m, iz = oz + nf * m;
        eX += Dy[m] * U(5, iy) - Dz[m] * U(4, iz) - Dx[m] * U(6, ix);
        eY += Dz[m] * U(3, iz) - Dx[m] * U(5, ix) - Dy[m] * U(6, iy);
        eZ += Dx[m] * U(4, ix) - Dy[m] * U(3, iy) - Dz[m] * U(6, iz);
        bX += Dz[m] * U(1, iz) - Dy[m] * U(2, iy) - Dx[m] * U(7, ix);
        bY += Dx[m] * U(2, ix) - Dz[m] * U(0, iz) - Dy[m] * U(7, iy);
        bZ += Dy[m] * U(0, iy) - Dx[m] * U(1, ix) - Dz[m] * U(7, iz);
        ps -= Dx[m] * U(0, ix) + Dy[m] * U(1, iy) + Dz[m] * U(2, iz);
        ph -= Dx[m] * U(3, ix) + Dy[m] * U(4, iy) + Dz[m] * U(5, iz);
        qq -= Dx[m] * J.dg(3)[eb + ix] + Dy[m] * J.dg(4)[eb + iy] + Dz[m] * J.dg(5)[eb + iz];
    }
    r[0] = eX; r[nn] = eY; r[2 * nn] = eZ; r[3 * nn] = bX; r[4 * nn] = bY; r[5 * nn] = bZ;
    r[6 * nn] = ps; r[7 * nn] = ph; r[8 * nn] = qq;
}

// What bounds it: the FP64 pipe (2 lanes a clock and SM; a warp instruction takes
// 16 clocks of an SM).  So the line contractions of the volume term, the filter and the
// indicator, 290 of 430 FP64 slots a thread, run on the integer pipes (fixed.cuh: a
// 32 x 32 -> 64 bit multiply-add takes one clock a warp, three of them replace an FMA);
// in the rest
// the work per node is what counts: five lift values per face node instead of nine,
// their sum into dU/dt axis by axis instead of node by node under divergence, no FP64
// comparisons, and the stage's G and currents from its solve (substep_implicit).
// Four CTAs an SM, whose barriers hide each other's, at 72 registers: J~ is not kept in
// shared memory but for its fixed-point form (three CTAs: 0.413 ms a substep of the
// current sheet against 0.402; two without spills: 3% slower than three).
// 4096 elements at P = 5, average of the substeps: 0.870 ms, 0.757 with less work per
// node, 0.551 with the volume term in integers, 0.493 with the indicator, 0.444 with the
// filter, 0.440 with four CTAs, 0.421 axis by axis with a scale for every variable and
// axis (a row of D is loaded once, 588 bytes of spills instead of 952).
template <int P, int SUB>
__global__ void __launch_bounds__(DGK<P>::NT, DGK<P>::CTAS) k_dg_substep(Dev d, SubArgs a) {
    using K = DGK<P>;
    constexpr int np1 = K::np1, nn = K::nn, nf = K::nf, NT = K::NT;
    extern __shared__ double sm[];
    double* sU = sm;                 // [9][nn]
    double* sR = sU + 9 * nn;        // [9][nn] dU/dt
    Fx* fU = (Fx*)(sR + 9 * nn);     // [12][nn] U and J~ in fixed point
    double* red = sR + 21 * nn;
    double* sD = red + 2;            // [3][np1][np1]: (d xi^a/d x^a) D
    Fx* fD = (Fx*)sD;
    __shared__ int s_flag;
    // largest words (fx_word) of U and J~, of the filter's variables, of |B~|
    __shared__ unsigned s_word[12], s_wordf[NV + 1];
    __shared__ int s_eq[NV], s_shift[3 * NV];   // exponents of the volume term's sums, shifts of their terms to them
    const Tables& T = *d.tab;
    const int tid = threadIdx.x;
    const bool act = tid < nn;
    const int i = tid % np1, j = (tid / np1) % np1, k = tid / (np1 * np1);
    const double w0inv = 1.0 / T.w0;
    const int nwork = d.counts[0];
    if (tid < 12) s_word[tid] = 0;
    __syncthreads();
    for (int w = blockIdx.x; w < nwork; w += gridDim.x) {
        const int e = d.dg_list[w];
        const int64_t eb = (int64_t)e * nn;
        const double sx = d.ijac[3 * e], sy = d.ijac[3 * e + 1], sz = d.ijac[3 * e + 2];
        double* r = sR + tid;
        unsigned word[12];
        double jx[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int v = 0; v < 12; ++v) {
            word[v] = 0;
            if (!act) continue;
            const double x = v < NV ? a.Uin.dg(v)[eb + tid] : a.J.dg(3 + v - NV)[eb + tid];
            if (v < NV) sU[v * nn + tid] = x;
            else jx[v - NV] = x;
            if (v != 8) word[v] = fx_word(x);   // q~ is not differentiated
        }
        fx_largest<12>(word, s_word);
        const double rows[3] = {T.Dabs * fabs(sx), T.Dabs * fabs(sy), T.Dabs * fabs(sz)};   // bound the rows' |D| sums
        int eD[3];
        bool fixed = true;
        for (int k = 0; k < 3; ++k) {
            eD[k] = (int)(fx_word(rows[k]) >> 20);
            fixed = fixed && eD[k] > 1023 - 60 && eD[k] < 1023 + 60;
        }
        __syncthreads();
        if (tid <= NV) s_wordf[tid] = 0;
#pragma unroll
        for (int v = 0; v < 12; ++v) fixed = fixed && fx_inside(s_word[v]);
        if (tid < NV) {
            int e[3];
            for (int k = 0; k < 3; ++k) e[k] = fx_exp(s_word[term_var(tid, k)]) + eD[k];
            const int top = max(e[0], max(e[1], e[2]));
            s_eq[tid] = top;
            for (int k = 0; k < 3; ++k) s_shift[3 * tid + k] = min(top - e[k], 63);
        }
        for (int t = tid; t < 3 * nf; t += NT) {
            const int k = t < nf ? 0 : (t < 2 * nf ? 1 : 2);
            const double D = (k == 0 ? sx : (k == 1 ? sy : sz)) * T.D[(t % nf) / np1][t % np1];
            if (fixed) fD[t] = fx_limbs(fx_from(D, k == 0 ? eD[0] : (k == 1 ? eD[1] : eD[2]), FX_BITS));
            else sD[t] = D;
        }
        if (act && fixed) {
#pragma unroll
            for (int v = 0; v < 12; ++v)
                if (v != 8) fU[v * nn + tid] = fx_limbs(fx_from(v < NV ? sU[v * nn + tid] : jx[v < NV ? 0 : v - NV], fx_exp(s_word[v]), FX_BITS));
        }
        __syncthreads();
        if (tid < 12) s_word[tid] = 0;
        if (act && fixed) {
            // Nine sums of three lines each: E~: curl B~ - grad psi~ - J~, B~: -curl E~ - grad phi~,
            // psi~: -div E~ + q~, phi~: -div B~, q~: -div J~; axis by axis, so that a row of D is
            // loaded once, every line at its own scale and shifted to its sum's
            long long acc[NV];
#pragma unroll
            for (int q = 0; q < NV; ++q) acc[q] = 0;
#pragma unroll
            for (int ax = 0; ax < 3; ++ax) {
                const int stride = ax == 0 ? 1 : (ax == 1 ? np1 : nf), c = ax == 0 ? i : (ax == 1 ? j : k);
                const Fx* line = fU + tid - c * stride;
                Fx Dr[np1];
#pragma unroll
                for (int m = 0; m < np1; ++m) Dr[m] = fD[ax * nf + np1 * c + m];
#pragma unroll
                for (int q = 0; q < NV; ++q) {
                    FxSum s;
#pragma unroll
                    for (int m = 0; m < np1; ++m) s.add(line[term_var(q, ax) * nn + m * stride], Dr[m]);
                    const long long t = s.top() >> s_shift[3 * q + ax];
                    acc[q] += term_neg(q, ax) ? -t : t;
                }
            }
            // units: 2^60 2^(e - 1022 - 60) 2^(eD - 1022 - 60)
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                double x = fx_double(acc[q], s_eq[q] - 2104);
                if (q < 3) x -= a.J.dg(q)[eb + tid];
                if (q == 6) x += sU[8 * nn + tid];
                r[q * nn] = x;
            }
        } else if (act) {
            volume_fp64<P>(a.J, eb, sU, sD, r);
        }
        // Lift, one thread per face node.  The jump (dU, dJ) to the exterior state
        // enters through the pairs (a, b, s) of flux_pair: with t = s (outward sign)
        // the correction of a is c = (t db - da) |grad xi|/(2 w0), that of b is -t c:
        // five values per face node.
        double cor[K::FR][5];
        int me[K::FR];
#pragma unroll
        for (int r = 0; r < K::FR; ++r) {
            const int t = tid + r * NT;
            if (t >= 6 * nf) break;
            const int f = t / nf, ab = t % nf, ta = ab % np1, tb = ab / np1;
            const int dd = f >> 1, s = f & 1;
            int t1, t2;
            face_axes(dd, t1, t2);
            int c[3];
            c[dd] = s ? P : 0;
            c[t1] = ta;
            c[t2] = tb;
            me[r] = node_index<P>(c[0], c[1], c[2]);
            double Ui[NV], Ue[NV], Je[3], xn[3];
            for (int v = 0; v < NV; ++v) Ui[v] = sU[v * nn + me[r]];
            if (d.nbr[e * 6 + f] < 0 && d.bc[e * 6 + f] == FFE_BC_STAR)
                for (int q = 0; q < 3; ++q) xn[q] = d.xyz_dg[(int64_t)q * d.ndg + eb + me[r]];
            dg_external_state<P>(d, a, e, f, ta, tb, Ui, xn, Ue, Je);
            const double jump = (dd == 0 ? Je[0] : (dd == 1 ? Je[1] : Je[2])) - a.J.dg(3 + dd)[eb + me[r]];
            const unsigned long long sg = s ? 0ULL : 0x8000000000000000ULL;
            const double scale = 0.5 * (dd == 0 ? sx : (dd == 1 ? sy : sz)) * w0inv;   // |grad xi^d| / (2 w0)
            for (int v = 0; v < NV; ++v) Ue[v] -= Ui[v];
            auto pair = [&](double da, double db, bool neg) { return scale * (flip(db, neg ? sg ^ 0x8000000000000000ULL : sg) - da); };
            auto pick = [&](double x, double y, double z) { return dd == 0 ? x : (dd == 1 ? y : z); };
            cor[r][0] = pair(pick(Ue[0], Ue[1], Ue[2]), Ue[6], false);
            cor[r][1] = pair(pick(Ue[3], Ue[4], Ue[5]), Ue[7], false);
            cor[r][2] = pair(pick(Ue[1], Ue[2], Ue[0]), pick(Ue[5], Ue[3], Ue[4]), false);
            cor[r][3] = pair(pick(Ue[2], Ue[0], Ue[1]), pick(Ue[4], Ue[5], Ue[3]), true);
            cor[r][4] = pair(Ue[8], jump, false);
        }
        // added axis by axis: edge and corner nodes lie on faces of several axes, so a
        // node-wise sum would diverge in every warp (54 FP64 slots a warp where 12 do)
        for (int dd = 0; dd < 3; ++dd) {
            __syncthreads();
#pragma unroll
            for (int r = 0; r < K::FR; ++r) {
                const int t = tid + r * NT;
                if (t < 2 * dd * nf || t >= 2 * (dd + 1) * nf) continue;
                const unsigned long long sg = (t / nf) & 1 ? 0ULL : 0x8000000000000000ULL;
#pragma unroll
                for (int pr = 0; pr < 5; ++pr) {
                    int va, vb;
                    bool neg;
                    flux_pair(dd, pr, va, vb, neg);
                    sR[va * nn + me[r]] -= cor[r][pr];
                    if (pr < 4) sR[vb * nn + me[r]] += flip(cor[r][pr], neg ? sg ^ 0x8000000000000000ULL : sg);
                }
            }
        }
        __syncthreads();
        double du[NV];
        if (act)
            for (int v = 0; v < NV; ++v) du[v] = sR[v * nn + tid];
        if (SUB == SUB_RHS) {
            if (act)
                for (int v = 0; v < NV; ++v) a.Fout.dg(v)[eb + tid] = du[v];
            __syncthreads();
            continue;
        }
        double u[NV];
        if (act) {
            if (SUB != SUB_C)
                for (int v = 0; v < NV; ++v) a.Fout.dg(v)[eb + tid] = du[v];
            substep_explicit(SUB, du, eb + tid, false, a, d.sk, u);
        }
        if (d.filter_on) {
            filter_element<P, NT>(T, act, sU, (long long*)fU, s_wordf, u);
        }
        // implicit part after the filter; G at the stage value: G_s = (U_s - R~_s)/(dt a)
        if (act) substep_implicit<SUB>(d, d.sk, a, eb + tid, false, u);
        bool flagged = false;
        if (d.tci_on) {
            const double mag = act ? sqrt(fma(u[5], u[5], fma(u[4], u[4], u[3] * u[3]))) : 0.0;
            const double ratio = indicator_ratio<P, NT>(T, act, mag, (long long*)fU, &s_wordf[NV], red);
            if (tid == 0) {
                int fl = ratio > d.thr_dg;
                if (fabs(ratio - d.thr_dg) <= 1e-12 * d.thr_dg) d.near_list[atomicAdd(&d.counts[3], 1) & 4095] = e;
                if (fl && take_fd_slot(d, e)) {
                    d.flag_list[atomicAdd(&d.counts[2], 1)] = e;
                    d.switched[e] = 1;
                } else {
                    fl = 0;
                }
                s_flag = fl;
            }
            __syncthreads();
            flagged = s_flag != 0;
        }
        if (!flagged && tid == 0) {
            atomicAdd(d.units, (unsigned long long)nn);
            atomicAdd(d.units + 2, 1ull);
        }
        if (!flagged && act) {
            bool bad = false;
            for (int v = 0; v < NV; ++v) {
                a.Uout.dg(v)[eb + tid] = u[v];
                bad |= !is_finite(u[v]);
            }
            if (bad) atomic_status(d, 1);
        }
        __syncthreads();
    }
}

template <int P>
static void dg_sub_dispatch(const Dev& d, int sub, const SubArgs& a, cudaStream_t st) {
    using K = DGK<P>;
    const int grid = d.dg_grid > 0 ? d.dg_grid : d.nsm * 4;
    switch (sub) {
        case SUB_A:
            cudaFuncSetAttribute(k_dg_substep<P, SUB_A>, cudaFuncAttributeMaxDynamicSharedMemorySize, K::SMEM);
            k_dg_substep<P, SUB_A><<<grid, K::NT, K::SMEM, st>>>(d, a);
            break;
        case SUB_B:
            cudaFuncSetAttribute(k_dg_substep<P, SUB_B>, cudaFuncAttributeMaxDynamicSharedMemorySize, K::SMEM);
            k_dg_substep<P, SUB_B><<<grid, K::NT, K::SMEM, st>>>(d, a);
            break;
        case SUB_C:
            cudaFuncSetAttribute(k_dg_substep<P, SUB_C>, cudaFuncAttributeMaxDynamicSharedMemorySize, K::SMEM);
            k_dg_substep<P, SUB_C><<<grid, K::NT, K::SMEM, st>>>(d, a);
            break;
        default:
            cudaFuncSetAttribute(k_dg_substep<P, SUB_RHS>, cudaFuncAttributeMaxDynamicSharedMemorySize, K::SMEM);
            k_dg_substep<P, SUB_RHS><<<grid, K::NT, K::SMEM, st>>>(d, a);
    }
    g_launch_counter += 1;
}

void launch_dg_substep(const Dev& d, int sub, Field Uin, Field J, Field un, Field F2, Field F3,
                       Field G1, Field G2, Field G3, Field G4, Field Fout, Field Uout, Field Gout, Field Jout,
                       cudaStream_t st) {
    SubArgs a{Uin, J, un, F2, F3, G1, G2, G3, G4, Fout, Uout, Gout, Jout};
    prof_begin(sub == SUB_RHS ? "dg_rhs" : "dg_substep", st);
    switch (d.P) {
        case 2: dg_sub_dispatch<2>(d, sub, a, st); break;
        case 3: dg_sub_dispatch<3>(d, sub, a, st); break;
        case 4: dg_sub_dispatch<4>(d, sub, a, st); break;
        case 5: dg_sub_dispatch<5>(d, sub, a, st); break;
        case 6: dg_sub_dispatch<6>(d, sub, a, st); break;
        default: break;
    }
    prof_end(st);
}

// ---------------------------------------------------------------------------
// Indicator ratio of the DG data of every element (diagnostic entry point).
__global__ void k_tci_ratio(Dev d, const double* Udg, double* ratio) {
    __shared__ double su[MAXNP * MAXNP * MAXNP * 3];
    __shared__ double red[2];
    for (int e = blockIdx.x; e < d.E; e += gridDim.x) {
        const ES es = esz(d, e);
        const Tables& T = d.tabs[es.P];
        const int np1 = es.np1, nn = es.nn;
        for (int t = threadIdx.x; t < nn; t += blockDim.x) {
            const int64_t p = (int64_t)e * d.nn + t;
            const double bx = Udg[3 * d.ndg + p], by = Udg[4 * d.ndg + p], bz = Udg[5 * d.ndg + p];
            su[t] = sqrt(fma(bz, bz, fma(by, by, bx * bx)));
        }
        __syncthreads();
        for (int t = threadIdx.x; t < nn; t += blockDim.x) {
            const int i = t % np1, j = (t / np1) % np1, k = t / (np1 * np1);
            double acc = 0.0;
            for (int m = 0; m < np1; ++m) acc = fma(T.Pi[i][m], su[m + np1 * (j + np1 * k)], acc);
            su[nn + t] = acc;
        }
        __syncthreads();
        for (int t = threadIdx.x; t < nn; t += blockDim.x) {
            const int i = t % np1, j = (t / np1) % np1, k = t / (np1 * np1);
            double acc = 0.0;
            for (int m = 0; m < np1; ++m) acc = fma(T.Pi[j][m], su[nn + i + np1 * (m + np1 * k)], acc);
            su[2 * nn + t] = acc;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double num = 0.0, den = 0.0;
            for (int t = 0; t < nn; ++t) {
                const int i = t % np1, j = (t / np1) % np1, k = t / (np1 * np1);
                double acc = 0.0;
                for (int m = 0; m < np1; ++m) acc = fma(T.Pi[k][m], su[2 * nn + i + np1 * (j + np1 * m)], acc);
                const double uh = su[t] - acc;
                num += uh * uh;
                den += su[t] * su[t];
            }
            red[0] = den > 0.0 ? sqrt(num / den) : 0.0;
            ratio[e] = red[0];
        }
        __syncthreads();
    }
}

void launch_tci_ratio(const Dev& d, const double* Udg, double* ratio, cudaStream_t st) {
    prof_begin("tci_ratio", st);
    k_tci_ratio<<<d.nsm * 4, 128, 0, st>>>(d, Udg, ratio);
    prof_end(st);
    g_launch_counter += 1;
}

// ---------------------------------------------------------------------------
// Pointwise constraint diagnostics of a state (flat metric, densitised fields):
// per block max |E~.B~|, min (B~^2 - E~^2), max |psi~|, max |phi~| over the DG
// nodes of DG elements and the cells of FD elements.
__device__ __forceinline__ void cons_point(const Field& U, bool fd, int64_t p, double* r) {
    double u[8];
    for (int v = 0; v < 8; ++v) u[v] = fd ? U.fd(v)[p] : U.dg(v)[p];
    const double EB = fma(u[2], u[5], fma(u[1], u[4], u[0] * u[3]));
    const double D = fma(u[5], u[5], fma(u[4], u[4], u[3] * u[3])) - fma(u[2], u[2], fma(u[1], u[1], u[0] * u[0]));
    r[0] = fmax(r[0], fabs(EB));
    r[1] = fmin(r[1], D);
    r[2] = fmax(r[2], fabs(u[6]));
    r[3] = fmax(r[3], fabs(u[7]));
}

__global__ void k_constraints(Dev d, Field U, double* part) {
    __shared__ double sr[4][256];
    double r[4] = {0.0, 1.0e308, 0.0, 0.0};
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p = tid; p < d.ndg; p += stride) {
        const int e = (int)(p / d.nn);
        if (d.mask[e] == 0 && (int)(p % d.nn) < esz(d, e).nn) cons_point(U, false, p, r);
    }
    for (int64_t p = tid; p < d.nfd; p += stride) {
        const int sl = (int)(p / d.ncell);
        const int e = d.slot_elem ? d.slot_elem[sl] : sl;
        if (e >= 0 && d.mask[e] == 1 && (int)(p % d.ncell) < esz(d, e).ncell) cons_point(U, true, p, r);
    }
    for (int i = 0; i < 4; ++i) sr[i][threadIdx.x] = r[i];
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) {
            sr[0][threadIdx.x] = fmax(sr[0][threadIdx.x], sr[0][threadIdx.x + o]);
            sr[1][threadIdx.x] = fmin(sr[1][threadIdx.x], sr[1][threadIdx.x + o]);
            sr[2][threadIdx.x] = fmax(sr[2][threadIdx.x], sr[2][threadIdx.x + o]);
            sr[3][threadIdx.x] = fmax(sr[3][threadIdx.x], sr[3][threadIdx.x + o]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int i = 0; i < 4; ++i) part[4 * blockIdx.x + i] = sr[i][0];
}

void launch_constraints(const Dev& d, Field U, double* part, int blocks, cudaStream_t st) {
    k_constraints<<<blocks, 256, 0, st>>>(d, U, part);
    g_launch_counter += 1;
}

// L2 error norm of Sec. IV.B.1 (Table II), sum part: per block the sum over
// the DG nodes of DG elements and the cells of FD elements of
// sum_{v0 <= v < v0 + nv} (U_v - R_v)^2, accumulated per thread in index
// order and reduced by a fixed tree (deterministic for a fixed grid).
__global__ void k_l2_err(Dev d, Field U, Field R, int v0, int nv, double* part) {
    __shared__ double sr[256];
    double acc = 0.0;
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p = tid; p < d.ndg; p += stride) {
        const int e = (int)(p / d.nn);
        if (d.mask[e] == 0 && (int)(p % d.nn) < esz(d, e).nn)
            for (int v = v0; v < v0 + nv; ++v) {
                const double df = U.dg(v)[p] - R.dg(v)[p];
                acc = fma(df, df, acc);
            }
    }
    for (int64_t p = tid; p < d.nfd; p += stride) {
        const int sl = (int)(p / d.ncell);
        const int e = d.slot_elem ? d.slot_elem[sl] : sl;
        if (e >= 0 && d.mask[e] == 1 && (int)(p % d.ncell) < esz(d, e).ncell)
            for (int v = v0; v < v0 + nv; ++v) {
                const double df = U.fd(v)[p] - R.fd(v)[p];
                acc = fma(df, df, acc);
            }
    }
    sr[threadIdx.x] = acc;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sr[threadIdx.x] += sr[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sr[0];
}

void launch_l2_err(const Dev& d, Field U, Field R, int v0, int nv, double* part, int blocks, cudaStream_t st) {
    k_l2_err<<<blocks, 256, 0, st>>>(d, U, R, v0, nv, part);
    g_launch_counter += 1;
}

}  // namespace ffe
