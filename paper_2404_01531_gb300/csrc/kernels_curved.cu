// DG substep on curved elements (cubed-sphere shells), flat or Kerr-Schild metric.
//
// Per element (one CTA, one thread per LGL node) the chain-rule strong form
//   dU/dt = - sum_k sum_j (d xi^k/d x^j)_n (D_k F^j)_n + S
//           - sum_faces (|grad xi^d|_gamma / w0) (F*.n^ - F_int.n^)
// with F^j the physical fluxes at the nodes (Sec. II.A), the inverse Jacobian
// of the element map at each node, the Rusanov flux with lambda = alpha +
// |beta.n^|, then the same stage order as the box kernel (explicit part,
// filter, stiff solve, clamp, indicator).  The stiff solve, clamp and indicator
// use the gamma inner product.
#include "dgfilter.cuh"
#include "dgtci.cuh"
#include "ffe_internal.h"
#include "physics.cuh"
#include "physics_gen.cuh"
#include "shellmap.cuh"
#include "stage.cuh"

namespace ffe {

template <int P, bool KS>
struct DGC {
    static constexpr int np1 = P + 1;
    static constexpr int nn = np1 * np1 * np1;
    static constexpr int nf = np1 * np1;
    static constexpr int NT = ((nn + 31) / 32) * 32;
    static constexpr int FR = (6 * nf + NT - 1) / NT;   // face nodes per thread
    // CTAs per SM the registers are bounded for (see k_dg_curved)
    static constexpr int CTAS = NT <= 128 ? (KS ? 3 : 4) : 2;
    // shared doubles: U[9][nn] (later the filter's buffer) | J[3][nn] | fixed point:
    // U and J [12][nn], Kerr-Schild: F[27][nn] as doubles, then in fixed point (later the
    // filter's and the indicator's fields) | dU/dt[9][nn] | red[2] and the flag
    static constexpr int NS = KS ? 30 : 15;
    static constexpr int SMEM = ((18 + NS) * nn + 3) * 8;
};

// neighbour's node for my face node (ta, tb) of face f
template <int P>
__device__ __forceinline__ void nbr_node(const Dev& d, int e, int f, int ta, int tb, int c[3]) {
    const int f2 = d.nbr_face[e * 6 + f], d2 = f2 >> 1;
    const int u1 = d2 == 0 ? 1 : 0, u2 = d2 == 2 ? 1 : 2;
    int a2, b2;
    orient_map(d.orient[e * 6 + f], P + 1, ta, tb, a2, b2);
    c[d2] = (f2 & 1) ? P : 0;
    c[u1] = a2;
    c[u2] = b2;
}

// Outward unit normal (lower index) at face node ab of face f, |grad xi|_gamma / (2 w0)
// and lambda = alpha + |beta.n| (Dev::fgeo, k_face_geo)
__device__ __forceinline__ const double* face_geo(const Dev& d, int e, int f, int ab) {
    return d.fgeo + (((int64_t)e * 6 + f) * NFG) * d.np1 * d.np1 + ab;
}

__global__ void k_face_geo(Dev d, double* out) {
    const int nfm = d.np1 * d.np1;
    const int64_t total = (int64_t)d.E * 6 * nfm;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int ab = (int)(t % nfm), f = (int)((t / nfm) % 6), e = (int)(t / (6 * nfm));
        const ES es = esz(d, e);
        const int np1 = es.np1;
        if (ab >= np1 * np1) continue;
        const int dd = f >> 1, s = f & 1;
        int c[3];
        c[dd] = s ? es.P : 0;
        c[dd == 0 ? 1 : 0] = ab % np1;
        c[dd == 2 ? 1 : 2] = ab / np1;
        const int64_t p = (int64_t)e * d.nn + c[0] + np1 * (c[1] + np1 * c[2]);
        const double w0inv = 1.0 / d.tabs[es.P].w0;
        double nl[3], nu[3], lam = 1.0;
        for (int i = 0; i < 3; ++i) nu[i] = nl[i] = (s ? 1.0 : -1.0) * d.geo[(int64_t)(3 * dd + i) * d.ndg + p];
        PM m;
        if (d.ks) {
            load_pm(d.met, d.ndg, p, m);
            for (int i = 0; i < 3; ++i)
                nu[i] = fma(m.gu[sym3(i, 0)], nl[0], fma(m.gu[sym3(i, 1)], nl[1], m.gu[sym3(i, 2)] * nl[2]));
        }
        const double norm = sqrt(d3(nu, nl)), inrm = 1.0 / norm;
        for (int i = 0; i < 3; ++i) nl[i] *= inrm;
        if (d.ks) lam = m.a + fabs(d3(m.b, nl));
        double* o = out + (((int64_t)e * 6 + f) * NFG) * nfm + ab;
        for (int i = 0; i < 3; ++i) o[i * nfm] = nl[i];
        o[3 * nfm] = 0.5 * norm * w0inv;
        o[4 * nfm] = lam;
    }
}

void launch_face_geo(const Dev& d, double* out, cudaStream_t st) {
    k_face_geo<<<d.nsm * 8, 256, 0, st>>>(d, out);
    g_launch_counter += 1;
}

// Exterior state at face node (face f, tangential ta, tb; node p, interior state Ui,
// outward unit normal nl) and its current J~; false where the current is J~(Ue)
template <int P, bool KS>
__device__ __forceinline__ bool curved_external(const Dev& d, const SubArgs& a, int e, int f, int ta, int tb, int64_t p,
                                                const double* Ui, const double* nl, double* Ue, double* Je) {
    constexpr int np1 = P + 1, nf = np1 * np1;
    const int nb = d.nbr[e * 6 + f];
    if (nb >= 0) {
        int cn[3];
        nbr_node<P>(d, e, f, ta, tb, cn);
        if (d.mask[nb] == 0) {
            const int64_t q = (int64_t)nb * d.nn + cn[0] + np1 * (cn[1] + np1 * cn[2]);
            for (int v = 0; v < NV; ++v) Ue[v] = a.Uin.dg(v)[q];
            if (!KS)
                for (int k = 0; k < 3; ++k) Je[k] = a.J.dg(3 + k)[q];
            return !KS;
        }
        // FD->DG projection (6-point stencils) of the neighbour's cells and of
        // their current J~ (the current of a projected state would carry its
        // projection error in E~.B~ amplified by eta into the q~ flux), from the face
        // traces face_trace left for it, indexed along the neighbour's own face axes
        const int f2 = d.nbr_face[e * 6 + f], d2 = f2 >> 1;
        const int u1 = d2 == 0 ? 1 : 0, u2 = d2 == 2 ? 1 : 2;
        const int nfm = d.np1 * d.np1;
        const double* tr = d.ftr + ((int64_t)fd_slot_of(d, nb) * 6 + f2) * 12 * nfm + cn[u1] + np1 * cn[u2];
        for (int v = 0; v < NV; ++v) Ue[v] = tr[v * nfm];
        for (int q = 0; q < 3; ++q) Je[q] = tr[(NV + q) * nfm];
        return true;
    }
    const int kind = d.bc[e * 6 + f];
    if (kind == FFE_BC_DIRICHLET) {
        const double* src = d.bdg + (int64_t)d.bface[e * 6 + f] * NV * nf;
        for (int v = 0; v < NV; ++v) Ue[v] = src[v * nf + ta + np1 * tb];
    } else if (kind == FFE_BC_NO_INCOMING) {
        if (KS) {
            PM mf;
            load_pm(d.met, d.ndg, p, mf);
            bc_no_incoming_gen(Ui, mf, nl, Ue);
        } else {
            bc_no_incoming_flat(Ui, nl, Ue);
        }
    } else if (kind == FFE_BC_OUTFLOW) {
        for (int v = 0; v < NV; ++v) Ue[v] = Ui[v];
    } else {
        double xn[3];
        for (int q = 0; q < 3; ++q) xn[q] = d.xyz_dg[(int64_t)q * d.ndg + p];
        bc_star_flat(Ui, xn, omega_of(d, e), Ue);
    }
    return false;
}

// n_j F^j of the flat flux at a jump (dU, dJ)
__device__ __forceinline__ void flux_normal_flat(const double* n, const double* U, const double* J, double* o) {
    const double *E = U, *B = U + 3;
    o[0] = fma(n[2], B[1], fma(n[1], -B[2], n[0] * U[6]));
    o[1] = fma(n[2], -B[0], fma(n[1], U[6], n[0] * B[2]));
    o[2] = fma(n[2], U[6], fma(n[1], B[0], n[0] * -B[1]));
    o[3] = fma(n[2], -E[1], fma(n[1], E[2], n[0] * U[7]));
    o[4] = fma(n[2], E[0], fma(n[1], U[7], n[0] * -E[2]));
    o[5] = fma(n[2], U[7], fma(n[1], -E[0], n[0] * E[1]));
    o[6] = fma(n[2], E[2], fma(n[1], E[1], n[0] * E[0]));
    o[7] = fma(n[2], B[2], fma(n[1], B[1], n[0] * B[0]));
    o[8] = fma(n[2], J[2], fma(n[1], J[1], n[0] * J[0]));
}

// n_j F^j with the metric (flux_gen contracted with n)
__device__ __forceinline__ void flux_normal_gen(const double* n, const PM& m, const double* U, const double* J, double* o) {
    double El[3], Bl[3], nu[3];
    lowr(m, U, El);
    lowr(m, U + 3, Bl);
    const double bn = d3(m.b, n), ia = m.a / m.sg;
    for (int i = 0; i < 3; ++i)
        nu[i] = m.a * fma(m.gu[sym3(i, 0)], n[0], fma(m.gu[sym3(i, 1)], n[1], m.gu[sym3(i, 2)] * n[2]));
    for (int i = 0; i < 3; ++i) {
        const int j = i == 2 ? 0 : i + 1, k = i == 0 ? 2 : i - 1;   // [ijk] n_j B_k = n_j B_k - n_k B_j, (i, j, k) cyclic
        o[i] = fma(-bn, U[i], fma(nu[i], U[6], -ia * fma(n[j], Bl[k], -n[k] * Bl[j])));
        o[3 + i] = fma(-bn, U[3 + i], fma(nu[i], U[7], ia * fma(n[j], El[k], -n[k] * El[j])));
    }
    o[6] = fma(-bn, U[6], m.a * d3(n, U));
    o[7] = fma(-bn, U[7], m.a * d3(n, U + 3));
    o[8] = fma(-bn, U[8], d3(n, J));
}

// One element of order P processed by a block of NT threads (NT >= (P+1)^3).
// s_word [27, flat 12]: the largest words (fx_word) of the volume term's fields, zero on
// entry and on return; s_wordf [NV + 1]: of the filter's and of |B~|.
template <int P, int NT, int SUB, bool KS>
__device__ __forceinline__ void dg_curved_elem(const Dev& d, const SubArgs& a, int e, double* sm, unsigned* s_word,
                                               unsigned* s_wordf) {
    using K = DGC<P, KS>;
    constexpr int np1 = K::np1, nn = K::nn, nf = K::nf;
    double* sU = sm;                 // [9][nn]
    double* sJ = sU + 9 * nn;        // [3][nn] J~ (full)
    double* sF = sJ + 3 * nn;        // fixed point [12][nn]; Kerr-Schild: [3][9][nn] F^j
    Fx* fF = (Fx*)sF;
    double* sR = sJ + K::NS * nn;    // [9][nn] dU/dt
    double* red = sR + 9 * nn;
    const Tables& T = d.tabs[P];
    const int tid = threadIdx.x;
    const bool act = tid < nn;
    const int ci[3] = {tid % np1, (tid / np1) % np1, tid / (np1 * np1)};
    const int64_t eb = (int64_t)e * d.nn;
    const double dt = dt_of(d, e);
    // Fields of the volume term's contractions, each at its own scale (fixed.cuh): U and J~,
    // or on the Kerr-Schild background the 27 fluxes.
    constexpr int NB = KS ? 27 : 12;
    unsigned word[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) word[b] = 0;
    if (act) {
#pragma unroll
        for (int v = 0; v < (KS ? NV : 12); ++v) {
            const double x = v < NV ? a.Uin.dg(v)[eb + tid] : a.J.dg(3 + v - NV)[eb + tid];
            sU[v * nn + tid] = x;
            if (!KS && v != 8) word[v] = fx_word(x);   // q~ is not differentiated
        }
        if (KS) {
            PM m;
            load_pm(d.met, d.ndg, eb + tid, m);
            double u[NV], jd[3], jf[3], F[3][NV], S[NV];
            for (int v = 0; v < NV; ++v) u[v] = sU[v * nn + tid];
            current_gen(u, m, d.eta, jd, jf);
            flux_gen(u, jf, m, F);
            for (int i = 0; i < 3; ++i) sJ[i * nn + tid] = jf[i];
            for (int j = 0; j < 3; ++j)
                for (int v = 0; v < NV; ++v) {
                    sF[(j * NV + v) * nn + tid] = F[j][v];
                    word[(j * NV + v) % NB] = fx_word(F[j][v]);
                }
            sources_gen(u, jd, m, d.met, d.ndg, eb + tid, S);
            for (int v = 0; v < NV; ++v) sR[v * nn + tid] = S[v];
        }
    }
    fx_largest<NB>(word, s_word);
    __syncthreads();
    if (tid <= NV) s_wordf[tid] = 0;
    bool fixed = !d.fp64_lines;
#pragma unroll
    for (int b = 0; b < NB; ++b) fixed = fixed && fx_inside(s_word[b]);
    if (act && fixed) {
#pragma unroll
        for (int v = 0; v < NB; ++v)
            if (KS || v != 8) fF[v * nn + tid] = fx_limbs(fx_from((KS ? sF : sU)[v * nn + tid], fx_exp(s_word[v]), FX_BITS));
    }
    __syncthreads();
    if (act) {
        double du[NV];
        for (int v = 0; v < NV; ++v) du[v] = KS ? sR[v * nn + tid] : 0.0;
        // derivatives along axis k with R(v) = D_k of value v
        auto volume = [&](int k, auto R) {
            double g[3];
            for (int i = 0; i < 3; ++i) g[i] = d.geo[(int64_t)(3 * k + i) * d.ndg + eb + tid];
            if (KS) {
                for (int j = 0; j < 3; ++j)
#pragma unroll
                    for (int v = 0; v < NV; ++v) du[v] = fma(-g[j], R(j * NV + v), du[v]);
            } else {
                // flat metric: D_k F^j = +-D_k of one field (D_k is linear), so the
                // volume term is built from the reference derivatives R = D_k X of the
                // 11 fields X = E~, B~, psi~, phi~, J~ and the node's d xi^k/d x^j:
                //   E~: curl B~ - grad psi~,  B~: -curl E~ - grad phi~,
                //   psi~: -div E~,  phi~: -div B~,  q~: -div J~
                const double ka = g[0], kb = g[1], kc = g[2];
                double r;
                r = R(0);   // E0
                du[4] = fma(-kc, r, du[4]); du[5] = fma(kb, r, du[5]); du[6] = fma(-ka, r, du[6]);
                r = R(1);   // E1
                du[3] = fma(kc, r, du[3]); du[5] = fma(-ka, r, du[5]); du[6] = fma(-kb, r, du[6]);
                r = R(2);   // E2
                du[3] = fma(-kb, r, du[3]); du[4] = fma(ka, r, du[4]); du[6] = fma(-kc, r, du[6]);
                r = R(3);   // B0
                du[1] = fma(kc, r, du[1]); du[2] = fma(-kb, r, du[2]); du[7] = fma(-ka, r, du[7]);
                r = R(4);   // B1
                du[0] = fma(-kc, r, du[0]); du[2] = fma(ka, r, du[2]); du[7] = fma(-kb, r, du[7]);
                r = R(5);   // B2
                du[0] = fma(kb, r, du[0]); du[1] = fma(-ka, r, du[1]); du[7] = fma(-kc, r, du[7]);
                r = R(6);   // psi
                du[0] = fma(-ka, r, du[0]); du[1] = fma(-kb, r, du[1]); du[2] = fma(-kc, r, du[2]);
                r = R(7);   // phi
                du[3] = fma(-ka, r, du[3]); du[4] = fma(-kb, r, du[4]); du[5] = fma(-kc, r, du[5]);
                r = R(9);   // J0
                du[8] = fma(-ka, r, du[8]);
                r = R(10);  // J1
                du[8] = fma(-kb, r, du[8]);
                r = R(11);  // J2
                du[8] = fma(-kc, r, du[8]);
            }
        };
        if (fixed) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int stride = k == 0 ? 1 : (k == 1 ? np1 : np1 * np1);
                const int base = tid - ci[k] * stride;
                Fx Dk[np1];
                for (int mm = 0; mm < np1; ++mm) Dk[mm] = T.FxD[ci[k]][mm];
                volume(k, [&](int v) {
                    FxSum s;
#pragma unroll
                    for (int mm = 0; mm < np1; ++mm) s.add(Dk[mm], fF[v * nn + base + mm * stride]);
                    // units: 2^60 2^-fx_d 2^(e - 1022 - 60)
                    return fx_double(s.top(), fx_exp(s_word[v]) - 1022 - T.fx_d);
                });
            }
        } else {
#pragma unroll 1
            for (int k = 0; k < 3; ++k) {
                const int stride = k == 0 ? 1 : (k == 1 ? np1 : np1 * np1);
                const int base = tid - ci[k] * stride;
                volume(k, [&](int v) {
                    double acc = 0.0;
#pragma unroll (KS ? 1 : np1)
                    for (int mm = 0; mm < np1; ++mm)
                        acc = fma(T.D[ci[k]][mm], (KS ? sF : sU)[v * nn + base + mm * stride], acc);
                    return acc;
                });
            }
        }
        if (!KS) {
            for (int i = 0; i < 3; ++i) du[i] -= a.J.dg(i)[eb + tid];
            du[6] += sU[8 * nn + tid];
        }
        for (int v = 0; v < NV; ++v) sR[v * nn + tid] = du[v];
    }
    // lift: one thread per face node.  The flux at a fixed point is linear in
    // (U, J~): F(Ue) - F(Ui) = F(Ue - Ui, Je - Ji), contracted with the normal at once
    double cor[K::FR][NV];
    int me[K::FR];
#pragma unroll
    for (int r = 0; r < K::FR; ++r) {
        const int t = tid + r * NT;
        if (t >= 6 * nf) break;
        const int f = t / nf, ab = t % nf, ta = ab % np1, tb = ab / np1;
        const int dd = f >> 1;
        int c[3];
        c[dd] = (f & 1) ? P : 0;
        c[dd == 0 ? 1 : 0] = ta;
        c[dd == 2 ? 1 : 2] = tb;
        me[r] = c[0] + np1 * (c[1] + np1 * c[2]);
        const int64_t p = eb + me[r];
        const double* fg = face_geo(d, e, f, ab);
        const int nfm = d.np1 * d.np1;
        const double nl[3] = {fg[0], fg[nfm], fg[2 * nfm]}, sc = fg[3 * nfm];
        double Ui[NV], Ue[NV], Je[3];
        for (int v = 0; v < NV; ++v) Ui[v] = sU[v * nn + me[r]];
        const bool given = curved_external<P, KS>(d, a, e, f, ta, tb, p, Ui, nl, Ue, Je);
        if (KS) {
            PM mf;
            load_pm(d.met, d.ndg, p, mf);
            if (!given) {
                double jde[3];
                current_gen(Ue, mf, d.eta, jde, Je);
            }
            for (int v = 0; v < NV; ++v) Ue[v] -= Ui[v];
            for (int i = 0; i < 3; ++i) Je[i] -= sJ[i * nn + me[r]];
            flux_normal_gen(nl, mf, Ue, Je, cor[r]);
            const double lam = fg[4 * nfm];
            for (int v = 0; v < NV; ++v) cor[r][v] = sc * fma(-lam, Ue[v], cor[r][v]);
        } else {
            if (!given) {
                double jde[3];
                current_flat(Ue, d.eta, jde, Je);
            }
            for (int v = 0; v < NV; ++v) Ue[v] -= Ui[v];
            for (int i = 0; i < 3; ++i) Je[i] -= sJ[i * nn + me[r]];
            flux_normal_flat(nl, Ue, Je, cor[r]);
            for (int v = 0; v < NV; ++v) cor[r][v] = sc * (cor[r][v] - Ue[v]);
        }
    }
    // added axis by axis (edge and corner nodes lie on faces of several axes; see k_dg_substep)
    for (int dd = 0; dd < 3; ++dd) {
        __syncthreads();
        if (dd == 0 && tid < NB) s_word[tid] = 0;
#pragma unroll
        for (int r = 0; r < K::FR; ++r) {
            const int t = tid + r * NT;
            if (t < 2 * dd * nf || t >= 2 * (dd + 1) * nf) continue;
            for (int v = 0; v < NV; ++v) sR[v * nn + me[r]] -= cor[r][v];
        }
    }
    __syncthreads();
    double du[NV], u[NV];
    if (act)
        for (int v = 0; v < NV; ++v) du[v] = sR[v * nn + tid];
    if (SUB == SUB_RHS) {
        if (act)
            for (int v = 0; v < NV; ++v) a.Fout.dg(v)[eb + tid] = du[v];
        __syncthreads();
        return;
    }
    if (act) {
        if (SUB != SUB_C)
            for (int v = 0; v < NV; ++v) a.Fout.dg(v)[eb + tid] = du[v];
        substep_explicit(SUB, du, eb + tid, false, a, solve_k(d, e), u);
    }
    if (d.filter_on) {
        filter_element<P, NT>(T, act, sU, (long long*)sF, s_wordf, u);
    }
    // implicit part after the filter; G at the stage value: G_s = (U_s - R~_s)/(dt a)
    double mag = 0.0;
    if (act) {
        if (KS) {
            PM m;
            load_pm(d.met, d.ndg, eb + tid, m);
            if (SUB != SUB_C && !stiff_solve_gen(u, m, d, dt * IM_A)) atomic_status(d, 2);
            if (d.mode != FFE_RELAX) hard_clamp_gen(u, m);
            if (SUB != SUB_C) {
                double g[NG];
                implicit_G_gen(u, m, d, g);
                for (int c = 0; c < NG; ++c) a.Gout.dg(c)[eb + tid] = g[c];
            }
            if (d.tci_on) mag = bnorm_gen(u, m);
        } else {
            substep_implicit<SUB>(d, solve_k(d, e), a, eb + tid, false, u);
            if (d.tci_on) mag = sqrt(fma(u[5], u[5], fma(u[4], u[4], u[3] * u[3])));
        }
    }
    bool flagged = false;
    if (d.tci_on) {
        const double ratio = indicator_ratio<P, NT>(T, act, mag, (long long*)sF, s_wordf + NV, red);
        const double thr = d.thr_dgP[P];
        if (tid == 0) {
            int fl = ratio > thr;
            if (fabs(ratio - thr) <= 1e-12 * thr) d.near_list[atomicAdd(&d.counts[3], 1) & 4095] = e;
            if (fl && take_fd_slot(d, e)) {
                d.flag_list[atomicAdd(&d.counts[2], 1)] = e;
                d.switched[e] = 1;
            } else {
                fl = 0;
            }
            red[2] = fl;
        }
        __syncthreads();
        flagged = red[2] != 0.0;
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


// Persistent kernel over a DG work list of order-P elements (list, count in
// d.counts[ci]).  Bound by the FP64 pipe, as the box kernel (k_dg_substep): the
// contractions of the volume term (198 FP64 slots a node, 486 with the metric) and of
// the filter run on the integer pipes, J~ is read instead of formed again at the nodes
// and at every face node, the normals and |grad xi| are tabulated, the jump's flux is
// contracted with the normal at once (27 FMAs; with the general metric's flux and a
// constant flat metric it was 170 slots), and the face sums go axis by axis.  Two CTAs
// an SM at P = 5 (P <= 4: three or four), also with the metric, which had one and idled
// at its barriers.  7146 elements of orders 4 and 5: substep 0.97 -> 0.64 ms (1.42 before
// the work outside the contractions went down); Kerr-Schild, 1536 elements: 0.77 ->
// 0.48 ms.  Batched contexts launch each order's elements separately, in
// CTAs sized for that order (one kernel dispatching on the order would keep every
// order's registers live and spill).
template <int P, int SUB, bool KS>
__global__ void __launch_bounds__(DGC<P, KS>::NT, DGC<P, KS>::CTAS) k_dg_curved(Dev d, SubArgs a, const int* list, int ci) {
    extern __shared__ double sm[];
    __shared__ unsigned s_word[27], s_wordf[NV + 1];
    if (threadIdx.x < 27) s_word[threadIdx.x] = 0;
    __syncthreads();
    const int nwork = d.counts[ci];
    for (int w = blockIdx.x; w < nwork; w += gridDim.x)
        dg_curved_elem<P, DGC<P, KS>::NT, SUB, KS>(d, a, list[w], sm, s_word, s_wordf);
}

template <int P, bool KS, int SUB>
static void curved_launch(const Dev& d, const SubArgs& a, const int* list, int ci, int grid, cudaStream_t st) {
    using K = DGC<P, KS>;
    cudaFuncSetAttribute(k_dg_curved<P, SUB, KS>, cudaFuncAttributeMaxDynamicSharedMemorySize, K::SMEM);
    k_dg_curved<P, SUB, KS><<<grid, K::NT, K::SMEM, st>>>(d, a, list, ci);
    g_launch_counter += 1;
}

template <int P, bool KS, int SUB>
static void curved_dispatch_sub(const Dev& d, const SubArgs& a, cudaStream_t st) {
    const int grid = d.dg_grid > 0 ? d.dg_grid : d.nsm * 2;
    curved_launch<P, KS, SUB>(d, a, d.dg_list, 0, grid, st);
    // batches: the elements of orders P-1 and P-2, each in CTAs sized for their order
    if constexpr (P > 3) {
        if (d.dg_list_lo)
            curved_launch<P - 1, KS, SUB>(d, a, d.dg_list_lo, 6, d.dg_grid_lo > 0 ? d.dg_grid_lo : d.nsm * 4, st);
    }
    if constexpr (P > 4) {
        if (d.dg_list_lo2)
            curved_launch<P - 2, KS, SUB>(d, a, d.dg_list_lo2, 7, d.dg_grid_lo2 > 0 ? d.dg_grid_lo2 : d.nsm * 4, st);
    }
}

template <int P, bool KS>
static void curved_dispatch(const Dev& d, int sub, const SubArgs& a, cudaStream_t st) {
    switch (sub) {
        case SUB_A: curved_dispatch_sub<P, KS, SUB_A>(d, a, st); break;
        case SUB_B: curved_dispatch_sub<P, KS, SUB_B>(d, a, st); break;
        case SUB_C: curved_dispatch_sub<P, KS, SUB_C>(d, a, st); break;
        default: curved_dispatch_sub<P, KS, SUB_RHS>(d, a, st); break;
    }
}

void launch_dg_substep_curved(const Dev& d, int sub, Field Uin, Field J, Field un, Field F2, Field F3, Field G1,
                              Field G2, Field G3, Field G4, Field Fout, Field Uout, Field Gout, Field Jout,
                              cudaStream_t st) {
    SubArgs a{Uin, J, un, F2, F3, G1, G2, G3, G4, Fout, Uout, Gout, Jout};
    prof_begin(sub == SUB_RHS ? "dg_rhs_curved" : "dg_substep_curved", st);
    if (d.ks) {
        switch (d.P) {
            case 3: curved_dispatch<3, true>(d, sub, a, st); break;
            case 4: curved_dispatch<4, true>(d, sub, a, st); break;
            case 5: curved_dispatch<5, true>(d, sub, a, st); break;
            default: break;
        }
    } else {
        switch (d.P) {
            case 3: curved_dispatch<3, false>(d, sub, a, st); break;
            case 4: curved_dispatch<4, false>(d, sub, a, st); break;
            case 5: curved_dispatch<5, false>(d, sub, a, st); break;
            default: break;
        }
    }
    prof_end(st);
}

// Stages 1 and 2 at DG nodes with the Kerr-Schild metric (FD is flat-only).
__global__ void k_stage12_ks(Dev d, Field un, Field Ua, Field G1, Field G2) {
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const double dta = d.dt * IM_A;
    auto point = [&](const PM& m, double* u, double* g1, double* g2) {
        double U1[NV];
        for (int v = 0; v < NV; ++v) U1[v] = u[v];
        if (!stiff_solve_gen(U1, m, d, dta)) atomic_status(d, 2);
        if (d.mode != FFE_RELAX) hard_clamp_gen(U1, m);
        implicit_G_gen(U1, m, d, g1);
        u[0] = fma(-dta, g1[0], u[0]);
        u[1] = fma(-dta, g1[1], u[1]);
        u[2] = fma(-dta, g1[2], u[2]);
        u[6] = fma(-dta, g1[3], u[6]);
        u[7] = fma(-dta, g1[4], u[7]);
        if (!stiff_solve_gen(u, m, d, dta)) atomic_status(d, 2);
        if (d.mode != FFE_RELAX) hard_clamp_gen(u, m);
        implicit_G_gen(u, m, d, g2);
    };
    for (int64_t p = tid; p < d.ndg; p += stride) {
        if (d.mask[p / d.nn] != 0) continue;
        PM m;
        load_pm(d.met, d.ndg, p, m);
        double u[NV], g1[NG], g2[NG];
        for (int v = 0; v < NV; ++v) u[v] = un.dg(v)[p];
        point(m, u, g1, g2);
        for (int v = 0; v < NV; ++v) Ua.dg(v)[p] = u[v];
        for (int c = 0; c < NG; ++c) { G1.dg(c)[p] = g1[c]; G2.dg(c)[p] = g2[c]; }
    }
    // FD cells of the FD list, with the metric at the subcell centre
    const int64_t nfdq = (int64_t)d.counts[1] * d.ncell;
    for (int64_t q = tid; q < nfdq; q += stride) {
        const int e = d.fd_list[q / d.ncell];
        const int c = (int)(q % d.ncell);
        const int64_t p = fdb(d, e) + c;
        PM m;
        load_pm(d.metfd, (int64_t)d.E * d.ncell, (int64_t)e * d.ncell + c, m);
        double u[NV], g1[NG], g2[NG];
        for (int v = 0; v < NV; ++v) u[v] = un.fd(v)[p];
        point(m, u, g1, g2);
        for (int v = 0; v < NV; ++v) Ua.fd(v)[p] = u[v];
        for (int cg = 0; cg < NG; ++cg) { G1.fd(cg)[p] = g1[cg]; G2.fd(cg)[p] = g2[cg]; }
    }
}

void launch_stage12_ks(const Dev& d, Field un, Field Ua, Field G1, Field G2, cudaStream_t st) {
    prof_begin("stage12", st);
    k_stage12_ks<<<d.nsm * 8, 256, 0, st>>>(d, un, Ua, G1, G2);
    prof_end(st);
    g_launch_counter += 1;
}

}  // namespace ffe
