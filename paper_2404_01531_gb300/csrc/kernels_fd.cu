// FD-subcell kernels of libffe, Sec. III.C.2:
//   k_fd_fill  builds, per listed FD element, an extended block of 12 quantities
//       (U and J~) with 3 ghost layers per face;
//   k_fd_flux (boxes), k_fd_states (flat shells)  one thread per line of cells
//       and pair of quantities: WENO5-Z (point-value interpolation form, Z weights
//       with q = 2) or MP5 face states, Rusanov flux, optional 4th-order corrector
//       with cell-centred fluxes; k_fd_flux_ks  one thread per face;
//   k_fd_update  one thread per cell: flux difference, sources, IMEX stage;
//   k_rollback_project  DG -> FD projection of a flagged element's substep inputs;
//   k_fd2dg      end-of-step FD -> DG check with alpha' = alpha + 1 (Sec. III.C.3).
// Listed FD elements are processed in chunks of d.chunk so that the scratch
// (extended blocks, face fluxes) is bounded whatever the number of FD elements.
// Elements may have different orders (batched contexts): every size below is
// the element's own; the slot strides d.ncell / (d.nc+6)^3 / (d.nc+1) d.nc^2
// are those of the largest order.
#include "ffe_internal.h"
#include "physics.cuh"
#include "physics_gen.cuh"
#include "shellmap.cuh"
#include "stage.cuh"
#include "fd_common.cuh"

namespace ffe {

// ---------------------------------------------------------------------------
// The 12 quantities of a cell, all loads before the first store that follows: the
// compiler has to assume that a store to the extended block changes what the next
// load reads, and a load waits some 700 clocks (125 elements of a box: fill 72 -> 64 us).
__device__ __forceinline__ void load_cell(const Field& U, const Field& J, int64_t p, double* q) {
#pragma unroll
    for (int v = 0; v < NV; ++v) q[v] = U.fd(v)[p];
#pragma unroll
    for (int k = 0; k < 3; ++k) q[NV + k] = J.fd(3 + k)[p];
}

// The element's own cells, to the middle of its extended block.
__device__ __forceinline__ void fill_interior(const Dev& d, int wl, int e, const Field& U, const Field& J) {
    const ES s = esz(d, e);
    const int nc = s.nc, ne = nc + 2 * GH;
    const int64_t fb = fdb(d, e);
    for (int c = threadIdx.x; c < s.ncell; c += blockDim.x) {
        const int x = c % nc, y = (c / nc) % nc, z = c / (nc * nc);
        const int o = (x + GH) + ne * ((y + GH) + ne * (z + GH));
        double q[NQ];
        load_cell(U, J, fb + c, q);
        for (int v = 0; v < NQ; ++v) ext_at(d, v, wl)[o] = q[v];
    }
}

// Face trace of an FD element for a DG neighbour (Sec. III.C.2 interface): at
// every LGL node of face f, if its neighbour is on DG, the FD->DG projection
// (6-point stencils along each axis) of the element's cells, for U and for its
// current J~.  A DG element facing an FD neighbour reads its exterior state here
// instead of projecting 6 x 6 x 6 cells per face node itself (which left most of
// its block idle).  Layout: per FD slot [6 faces][12 quantities][np1max^2], face
// node index a + np1 b along the face's axes (axes_of of its normal).  One CTA per
// (element, face): the projection is sum-factorised -- normal direction straight
// from the 6 cell layers next to the face, then the two tangential ones through
// shared memory -- 6 (nc^2 + nc np1 + np1^2) FMAs per quantity instead of 216 per
// face node.  Ends with a barrier.
__device__ __forceinline__ void face_trace(const Dev& d, int e, int f, const Field& U, const Field& J, double* sm) {
    const int nb = d.nbr[e * 6 + f];
    if (nb < 0 || d.mask[nb] != 0) return;
    const ES es = esz(d, e);
    const int np1 = es.np1, nc = es.nc, nc2 = nc * nc, nfm = d.np1 * d.np1;
    const Tables& T = d.tabs[es.P];
    const int dd = f >> 1;
    int t1, t2;
    axes_of(dd, t1, t2);
    const int cn = (f & 1) ? es.P : 0;       // the face's LGL index along the normal
    const int lo = T.f2d_lo[cn];
    double* A = sm;                            // [12][nc (t2)][nc (t1)]
    double* B = A + NQ * nc2;                  // [12][nc (t2)][np1 (t1)]
    const int64_t base = fdb(d, e);
    const int cs[3] = {1, nc, nc2};
    for (int t = threadIdx.x; t < NQ * nc2; t += blockDim.x) {
        const int q = t / nc2, ab = t % nc2;
        const double* src = (q < NV ? U.fd(q) : J.fd(3 + q - NV)) + base + lo * cs[dd] + (ab % nc) * cs[t1] + (ab / nc) * cs[t2];
        double acc = 0.0;
        for (int m = 0; m < 6; ++m) acc = fma(T.F2D[cn][lo + m], src[m * cs[dd]], acc);
        A[t] = acc;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < NQ * nc * np1; t += blockDim.x) {
        const int q = t / (nc * np1), r = t % (nc * np1);
        const int b = r / np1, i = r % np1;
        const int li = T.f2d_lo[i];
        double acc = 0.0;
        for (int m = 0; m < 6; ++m) acc = fma(T.F2D[i][li + m], A[(q * nc + b) * nc + li + m], acc);
        B[t] = acc;
    }
    __syncthreads();
    double* dst = d.ftr + ((int64_t)fd_slot_of(d, e) * 6 + f) * NQ * nfm;
    for (int t = threadIdx.x; t < NQ * np1 * np1; t += blockDim.x) {
        const int q = t / (np1 * np1), r = t % (np1 * np1);
        const int j = r / np1, i = r % np1;
        const int lj = T.f2d_lo[j];
        double acc = 0.0;
        for (int m = 0; m < 6; ++m) acc = fma(T.F2D[j][lj + m], B[(q * nc + lj + m) * np1 + i], acc);
        dst[q * nfm + i + np1 * j] = acc;
    }
    __syncthreads();
}

// 6 stencil weights of entry i of a per-slot table
__device__ __forceinline__ const double* gi_w(const double* table, const Dev& d, int slot, int i) {
    const int per = table == d.gwn ? GH : (table == d.gwr ? d.nc : GH * d.nc);
    return table + 6 * ((int64_t)slot * per + i);
}

// One CTA per (chunk position, face or interior): fill the extended block; with
// traces, also the element's face traces (both only read U and J~).
//
// Ghosts inside a wedge and on boxes are the neighbour's cells, or a DG
// neighbour's polynomial at its own subcell centres: the neighbour's grid lines
// continue this element's.  Across a face between two cubed-sphere wedges they
// bend, and a ghost is the neighbour's data at the ghost centre of this element's
// grid continued past the face (Sec. III.C.1): 6-point Lagrange interpolation of
// its cells and of their current J~, or its polynomial.  The map is equiangular
// and the radius is shared, so layer g of ghosts lies on the neighbour's own
// layer g and on its own radial cell centres: only the coordinate along the edge
// differs, and by an amount that depends on (g, ta) alone.  So of the 6 x 6 x 6
// weights of the tensor stencil only 6 are not zero, up to residues of 1e-15 where
// the two centres' coordinates differ in the last bit (one layer in six): the host
// tabulates the three axes' weights (Dev::gwn, gwf, gwr), zero ones and residues are
// skipped -- the residues are kept (36 or 216 products) for the adjoint's
// recomputation, which keeps its bits, see k_fd_flux_faces -- and a DG neighbour's
// polynomial takes three sum-factorised contractions.  With the interior's copy in
// the same launch, two launches fewer; 300 elements of a shell 1.99 -> 0.20 ms
// (0.53 with the residues).
__global__ void k_fd_fill(Dev d, const int* list, int ci, int w0, Field U, Field J, bool residues, bool traces) {
    const int n = chunk_n(d, ci, w0);
    const unsigned long long skip = residues ? 0ULL : fbits(1e-10);   // weights up to this are skipped
    extern __shared__ double sm[];
    const int items = traces ? 13 : 7;
    for (int item = blockIdx.x; item < n * items; item += gridDim.x) {
        const int wl = item / items, f = item % items;
        const int e = list[w0 + wl];
        if (f == 6) {
            fill_interior(d, wl, e, U, J);
            continue;
        }
        if (f > 6) {
            face_trace(d, e, f - 7, U, J, sm);
            continue;
        }
        const int gsl = d.gislot ? d.gislot[e * 6 + f] : -1;   // a face between wedges: its weights
        const ES es = esz(d, e);
        const Tables& T = d.tabs[es.P];
        const int nc = es.nc, ne = nc + 2 * GH, np1 = es.np1, nn = es.nn;
        double* su = sm;                          // neighbour DG block [12][nn]: U and J~
        double* t1b = su + NQ * nn;               // [12][GH][np1][np1]
        double* t2b = t1b + NQ * GH * np1 * np1;  // [12][GH][np1][nc]
        const int dd = f >> 1, s = f & 1;
        int t1, t2;
        axes_of(dd, t1, t2);
        const int nb = d.nbr[e * 6 + f];
        const int nper = GH * nc * nc;  // ghost cells of this face
        auto ghost_offset = [&](int g, int ta, int tb) -> int64_t {
            int c[3];
            c[dd] = s ? nc + GH + g : GH - 1 - g;
            c[t1] = ta + GH;
            c[t2] = tb + GH;
            return c[0] + (int64_t)ne * (c[1] + (int64_t)ne * c[2]);
        };
        if (nb >= 0 && d.mask[nb] == 1) {
            const int f2 = d.nbr_face[e * 6 + f];
            const int d2 = f2 >> 1, s2 = f2 & 1;
            int u1, u2;
            axes_of(d2, u1, u2);
            const int o = d.orient[e * 6 + f];
            const int64_t nbase = fdb(d, nb);
            for (int t = threadIdx.x; t < nper; t += blockDim.x) {
                const int g = t / (nc * nc), ta = t % nc, tb = (t / nc) % nc;
                int a2, b2;
                orient_map(o, nc, ta, tb, a2, b2);
                int c[3];
                if (gsl >= 0) {
                    // stencil weights along the neighbour's axes: all but one of those
                    // across the edge are zero, or a rounding residue for some layers
                    const double *w[3] = {nullptr, nullptr, gi_w(d.gwr, d, gsl, b2)};
                    int st[3];
                    w[d2] = gi_w(d.gwn, d, gsl, g);
                    w[u1] = gi_w(d.gwf, d, gsl, g * nc + ta);
                    st[d2] = d.gsn[gsl * GH + g];
                    st[u1] = d.gst[gsl * GH * d.nc + g * nc + ta];
                    st[2] = d.gsr[gsl * d.nc + b2];
                    const int64_t og = ghost_offset(g, ta, tb);
                    const int64_t p = nbase + st[0] + nc * (st[1] + nc * st[2]);
                    double acc[NQ];
                    for (int v = 0; v < NQ; ++v) acc[v] = 0.0;
                    for (int cz = 0; cz < 6; ++cz) {
                        if (fmag(w[2][cz]) <= skip) continue;
                        for (int cy = 0; cy < 6; ++cy) {
                            const double wzy = w[2][cz] * w[1][cy];
                            if (fmag(w[1][cy]) <= skip) continue;
                            for (int cx = 0; cx < 6; ++cx) {
                                if (fmag(w[0][cx]) <= skip) continue;
                                const double wt = wzy * w[0][cx];
                                const int64_t q = p + cx + nc * (cy + nc * cz);
                                for (int v = 0; v < NV; ++v) acc[v] = fma(wt, U.fd(v)[q], acc[v]);
                                for (int k = 0; k < 3; ++k) acc[NV + k] = fma(wt, J.fd(3 + k)[q], acc[NV + k]);
                            }
                        }
                    }
                    for (int v = 0; v < NQ; ++v) ext_at(d, v, wl)[og] = acc[v];
                    continue;
                }
                c[d2] = s2 ? nc - 1 - g : g;
                c[u1] = a2;
                c[u2] = b2;
                const int64_t p = nbase + c[0] + nc * (c[1] + nc * c[2]);
                const int64_t og = ghost_offset(g, ta, tb);
                double q[NQ];
                load_cell(U, J, p, q);
                for (int v = 0; v < NQ; ++v) ext_at(d, v, wl)[og] = q[v];
            }
        } else if (nb >= 0) {
            // DG neighbour: its polynomial at its own subcell centres (DG -> FD), 3
            // layers, for U and for its nodal current J~ (the current of the
            // evaluated state would carry the interpolation error of E~.B~ times eta)
            const int f2 = d.nbr_face[e * 6 + f];
            const int d2 = f2 >> 1, s2 = f2 & 1;
            int u1, u2;
            axes_of(d2, u1, u2);
            const int o = d.orient[e * 6 + f];
            for (int t = threadIdx.x; t < NQ * nn; t += blockDim.x) {
                const int qv = t / nn;
                const int64_t pn = (int64_t)nb * d.nn + t % nn;
                su[t] = qv < NV ? U.dg(qv)[pn] : J.dg(3 + qv - NV)[pn];
            }
            __syncthreads();
            // contract the normal direction for the 3 layers
            for (int t = threadIdx.x; t < NQ * GH * np1 * np1; t += blockDim.x) {
                const int v = t / (GH * np1 * np1), r = t % (GH * np1 * np1);
                const int g = r / (np1 * np1), a1 = r % np1, a2 = (r / np1) % np1;
                const int cn = s2 ? nc - 1 - g : g;
                double acc = 0.0;
                for (int m = 0; m < np1; ++m) {
                    int c[3];
                    c[d2] = m;
                    c[u1] = a1;
                    c[u2] = a2;
                    acc = fma(T.P2F[cn][m], su[v * nn + c[0] + np1 * (c[1] + np1 * c[2])], acc);
                }
                t1b[t] = acc;
            }
            __syncthreads();
            for (int t = threadIdx.x; t < NQ * GH * nc * np1; t += blockDim.x) {
                const int v = t / (GH * nc * np1), r = t % (GH * nc * np1);
                const int g = r / (nc * np1), ta = r % nc, a2 = (r / nc) % np1;
                // along u1: at the neighbour's cell ta, or at ghost ta's own point
                const double* w = gsl >= 0 ? d.gwl + ((int64_t)gsl * GH * d.nc + g * nc + ta) * MAXNP : T.P2F[ta];
                double acc = 0.0;
                for (int m = 0; m < np1; ++m) acc = fma(w[m], t1b[((v * GH + g) * np1 + a2) * np1 + m], acc);
                t2b[t] = acc;
            }
            __syncthreads();
            for (int t = threadIdx.x; t < nper; t += blockDim.x) {
                const int g = t / (nc * nc), ta = t % nc, tb = (t / nc) % nc;
                int a2, b2;   // the neighbour's subcell (along u1, u2) under this ghost cell
                orient_map(o, nc, ta, tb, a2, b2);
                if (gsl >= 0) a2 = ta;
                const int64_t og = ghost_offset(g, ta, tb);
                for (int v = 0; v < NQ; ++v) {
                    double acc = 0.0;
                    for (int m = 0; m < np1; ++m) acc = fma(T.P2F[b2][m], t2b[((v * GH + g) * np1 + m) * nc + a2], acc);
                    ext_at(d, v, wl)[og] = acc;
                }
            }
            __syncthreads();
        } else {
            const int kind = d.bc[e * 6 + f];
            for (int t = threadIdx.x; t < nper; t += blockDim.x) {
                const int g = t / (nc * nc), ta = t % nc, tb = (t / nc) % nc;
                double u[NV], jd[3], jf[3];
                if (kind == FFE_BC_DIRICHLET) {
                    const double* src = d.bfd + (int64_t)d.bface[e * 6 + f] * NV * GH * d.nc * d.nc;
                    for (int v = 0; v < NV; ++v) u[v] = src[(v * GH + g) * nc * nc + ta + nc * tb];
                } else {
                    // state from the outermost interior cell of this column
                    int c[3];
                    c[dd] = s ? nc - 1 : 0;
                    c[t1] = ta;
                    c[t2] = tb;
                    const int64_t p = fdb(d, e) + c[0] + nc * (c[1] + nc * c[2]);
                    double ui[NV];
                    for (int v = 0; v < NV; ++v) ui[v] = U.fd(v)[p];
                    if (kind == FFE_BC_NO_INCOMING) {
                        double nrm[3] = {0.0, 0.0, 0.0};
                        nrm[dd] = s ? 1.0 : -1.0;
                        if (d.curved) {
                            // outward unit normal at the face point of this column
                            shell_face_normal(shell_pts(d, e, nc), dd, s ? nc : 0, ta, tb, nrm);
                            if (!s)
                                for (int q = 0; q < 3; ++q) nrm[q] = -nrm[q];
                        }
                        bc_no_incoming_flat(ui, nrm, u);
                    } else if (kind == FFE_BC_OUTFLOW) {
                        for (int v = 0; v < NV; ++v) u[v] = ui[v];
                    } else {
                        double x[3];
                        if (d.curved) {
                            // centre of the outermost cell of this column
                            double ij[3][3];
                            shell_cell(shell_pts(d, e, nc), c, ij, x);
                        } else {
                            for (int k = 0; k < 3; ++k)
                                x[k] = d.xyz_fd[(int64_t)k * d.xfd_n + (int64_t)e * d.ncell + (p - fdb(d, e))];
                        }
                        bc_star_flat(ui, x, omega_of(d, e), u);
                    }
                }
                if (d.ks) {
                    // Dirichlet ghosts only on this background: metric at the ghost centre
                    PM m;
                    load_pm(d.metgb + (int64_t)d.bface[e * 6 + f] * NPM * GH * d.nc * d.nc, (int64_t)GH * d.nc * d.nc,
                            (int64_t)g * nc * nc + ta + nc * tb, m);
                    current_gen(u, m, d.eta, jd, jf);
                } else {
                    current_flat(u, d.eta, jd, jf);
                }
                const int64_t og = ghost_offset(g, ta, tb);
                for (int v = 0; v < NV; ++v) ext_at(d, v, wl)[og] = u[v];
                for (int k = 0; k < 3; ++k) ext_at(d, NV + k, wl)[og] = jf[k];
            }
        }
    }
}

// Box elements: one thread per (chunk position, direction, flux pair, line of
// cells).  The FP64 pipe (2 lanes a clock and SM) is the limit, everything else
// is nearly free beside it, so the split is the one with the fewest FP64
// operations: a thread marches a line and gives both face values of every cell
// from one set of smoothness indicators (Weno5zLine), for the two quantities
// that a pair of flux components needs, so that the flux is formed in registers;
// the two components of J~ across the direction are not reconstructed.  At P = 5
// that is 308 FP64 operations per face, the indicators and weights hidden on the
// integer pipes (z_weights), against about 1100 of a thread per face: 384 elements
// 3.44 -> 1.84 ms with 610 of them; two steps of the 64x8x8 current sheet 14.8 -> 13.7
// ms from 610 to 530, 11.6 with the weights in integers, 10.4 with the indicators too
// (9.6 with all of the step as it is);
// MP5 on 125 elements 1.53 -> 0.41 ms.
template <int RECON>
__global__ void __launch_bounds__(64, 8) k_fd_flux(Dev d, const int* list, int ci, int w0) {
    const int n = chunk_n(d, ci, w0);
    const int nc = d.nc, nl = nc * nc;
    const int per = 3 * FLUX_PAIRS * nl;
    const int64_t total = (int64_t)n * per;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int wl = (int)(t / per), r = (int)(t % per), line = r % nl, kp = r / nl;
        const int k = kp / FLUX_PAIRS, pr = kp % FLUX_PAIRS;
        int a, b;
        bool neg;
        flux_pair(k, pr, a, b, neg);
        int64_t stride;
        const int64_t base = line_start(k, line % nc, line / nc, nc, stride);
        const unsigned long long sb = neg ? 0x8000000000000000ULL : 0ULL;
        double* fa = flux_at(d, k, a, wl) + line;
        double* fb = pr < 4 ? flux_at(d, k, b, wl) + line : nullptr;
        const bool corr = d.fd_corr;
        recon_lines<typename LineOf<RECON>::type>(ext_at(d, a, wl) + base, ext_at(d, b, wl) + base, stride, sb, nc, d.weno_eps,
                           [&](int m, double La, double Ra, double Sa, double Lb, double Rb, double Sb) {
                               double Fa, Fb;
                               rusanov_pair(La, Ra, Sa, Lb, Rb, Sb, corr, Fa, Fb);
                               fa[m * nl] = Fa;
                               if (fb) fb[m * nl] = __longlong_as_double((long long)(fbits(Fb) ^ sb));
                           });
    }
}

// Flat-metric shells: one thread per (chunk position, direction, pair of
// quantities, line).  All three physical flux components enter a face there,
//   F^j = (F^j(L) + F^j(R))/2 - n^_j (U_R - U_L)/2  (lambda = 1, n^ the unit normal),
// optional corrector per component.  They are linear in the face states, so the
// kernel stores G = (L + R)/2 of the 12 quantities -- with the corrector
// (2/3)(L + R) - (U_m + U_p)/6 -- and D = (U_R - U_L)/2 -- times 4/3 -- of the 9
// variables: F^j = F^j(G) - n^_j D, formed once per cell by k_fd_update instead
// of once per face (21 values a face instead of 27, no normals here): 300 elements
// 2.74 -> 1.77 ms at P = 5 (0.92 with indicators and weights in integers),
// k_fd_update 0.28 -> 0.25 ms.
template <int RECON>
__global__ void __launch_bounds__(64, 8) k_fd_states(Dev d, const int* list, int ci, int w0) {
    const int n = chunk_n(d, ci, w0);
    const int nlm = d.nc * d.nc;
    const int per = 3 * (NQ / 2) * nlm;
    const int64_t total = (int64_t)n * per;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int wl = (int)(t / per), r = (int)(t % per), line = r % nlm, kp = r / nlm;
        const int k = kp / (NQ / 2), a = kp % (NQ / 2), b = a + NQ / 2;
        const int nc = esz(d, list[w0 + wl]).nc, nl = nc * nc;
        if (line >= nl) continue;
        int64_t stride;
        const int64_t base = line_start(k, line % nc, line / nc, nc, stride);
        double* ga = fstate_at(d, k, a, wl) + line;
        double* gb = fstate_at(d, k, b, wl) + line;
        double* da = fstate_at(d, k, NQ + a, wl) + line;
        double* db = b < NV ? fstate_at(d, k, NQ + b, wl) + line : nullptr;
        const bool corr = d.fd_corr;
        const double c1 = corr ? 2.0 / 3.0 : 0.5;
        recon_lines<typename LineOf<RECON>::type>(ext_at(d, a, wl) + base, ext_at(d, b, wl) + base, stride, 0ULL, nc, d.weno_eps,
                           [&](int m, double La, double Ra, double Sa, double Lb, double Rb, double Sb) {
                               double Ga = c1 * (La + Ra), Gb = c1 * (Lb + Rb);
                               if (corr) {
                                   Ga = fma(-1.0 / 6.0, Sa, Ga);
                                   Gb = fma(-1.0 / 6.0, Sb, Gb);
                               }
                               ga[m * nl] = Ga;
                               gb[m * nl] = Gb;
                               da[m * nl] = c1 * (Ra - La);
                               if (db) db[m * nl] = c1 * (Rb - Lb);
                           });
    }
}

// Flat shells, forward recomputation of the adjoint: one thread per face, all
// three flux components there.  A reverse step amplifies the rounding of the
// stages it is linearised at by up to 1e9 (J~ carries eta times the rounding of
// E~.B~, and the WENO5-Z weights' derivatives carry J~'s differences): inputs
// moved by one rounding move single entries of lambda_n by 7e-7 of their size.  So
// gradients stay comparable from one version to the next only if the
// recomputed stages keep their bits, and this kernel keeps the order of operations
// of a thread per face (k_fd_states: 1.5 times faster, different last bits).
__global__ void __launch_bounds__(128, 4) k_fd_flux_faces(Dev d, const int* list, int ci, int w0) {
    const int n = chunk_n(d, ci, w0);
    const int64_t nfc = nface(d);
    const int64_t total = (int64_t)n * 3 * nfc;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        const int wl = (int)(q / (3 * nfc));
        const int k = (int)((q / nfc) % 3);
        const int64_t fi = q % nfc;
        const int e = list[w0 + wl];
        const int nc = esz(d, e).nc;
        int m, ta, tb;
        if (!face_coords(fi, nc, m, ta, tb)) continue;
        double UL[NQ], UR[NQ], Um[NQ], Up[NQ];
        int64_t stride;
        int64_t base = line_start(k, ta, tb, nc, stride);   // sets stride
        base += m * stride;
        for (int qq = 0; qq < NQ; ++qq) {
            const double* src = ext_at(d, qq, wl) + base;
            const double v0 = src[0], v1 = src[stride], v2 = src[2 * stride];
            const double v3 = src[3 * stride], v4 = src[4 * stride], v5 = src[5 * stride];
            weno5z_pair(v0, v1, v2, v3, v4, v5, d.weno_eps, UL[qq], UR[qq]);
            Um[qq] = v2;
            Up[qq] = v3;
        }
        double nh[3];
        shell_face_normal(shell_pts(d, e, nc), k, m, ta, tb, nh);
        // the flat flux is linear in (U, J~): (F^j(L) + F^j(R))/2 = F^j((UL + UR)/2),
        // and the corrector's F(Um) + F(Up) = F(Um + Up)
        double hS[NQ], dU[NV], Sm[NQ];
        for (int qq = 0; qq < NQ; ++qq) hS[qq] = 0.5 * (UL[qq] + UR[qq]);
        for (int v = 0; v < NV; ++v) dU[v] = UR[v] - UL[v];
        if (d.fd_corr)
            for (int qq = 0; qq < NQ; ++qq) Sm[qq] = Um[qq] + Up[qq];
        for (int j = 0; j < 3; ++j) {
            double Fh[NV], Fs[NV];
            flux_dir_flat(hS, hS + NV, j, Fh);
            const double hn = -0.5 * nh[j];
            for (int v = 0; v < NV; ++v) Fs[v] = fma(hn, dU[v], Fh[v]);
            if (d.fd_corr) {
                double Fm[NV];
                flux_dir_flat(Sm, Sm + NV, j, Fm);
                for (int v = 0; v < NV; ++v) Fs[v] = fma(-1.0 / 6.0, Fm[v], (4.0 / 3.0) * Fs[v]);
            }
            for (int v = 0; v < NV; ++v) flux_at_c(d, k, j, v, wl)[face_index(nc, m, ta, tb)] = Fs[v];
        }
    }
}

// 12 left/right values of one face from the extended block
template <int RECON>
__device__ __forceinline__ void reconstruct(const Dev& d, int wl, int k, int m, int ta, int tb, int nc,
                                            double* UL, double* UR) {
    int64_t stride;
    int64_t base = line_start(k, ta, tb, nc, stride);   // sets stride
    base += m * stride;
    for (int qq = 0; qq < NQ; ++qq) {
        const double* src = ext_at(d, qq, wl) + base;
        typename LineOf<RECON>::type A;
        double none;
        A.init(src[0], src[stride], src[2 * stride], src[3 * stride], d.weno_eps);
        A.template cell<false, true>(src[4 * stride], none, UL[qq]);
        A.template cell<true, false>(src[5 * stride], UR[qq], none);
    }
}

// Kerr-Schild variant (Sec. III.C.2 on a curved background): the metric at
// the face point from Dev::metff; the unit normal n_l = d_l xi^k / |d xi^k|_gamma;
// Rusanov with lambda = alpha + |beta^l n_l| and the dissipation along
// n^j = gamma^jl n_l:
//   F^j = (F^j(L) + F^j(R))/2 - lambda n^j (U_R - U_L)/2,
// where the flux at a fixed point is linear in (U, J~), so its average is the
// flux of the averaged states.  No corrector (it is defined for Cartesian
// meshes; FFE_ENOTIMPL at creation).
template <int RECON>
__global__ void __launch_bounds__(128, 4) k_fd_flux_ks(Dev d, const int* list, int ci, int w0) {
    const int n = chunk_n(d, ci, w0);
    const int64_t nfc = nface(d);
    const int64_t total = (int64_t)n * 3 * nfc;
    const int64_t nfaces = (int64_t)d.E * nfc;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        const int wl = (int)(q / (3 * nfc));
        const int k = (int)((q / nfc) % 3);
        const int64_t fi = q % nfc;
        const int e = list[w0 + wl];
        const int nc = esz(d, e).nc;
        int m, ta, tb;
        if (!face_coords(fi, nc, m, ta, tb)) continue;
        double UL[NQ], UR[NQ];
        reconstruct<RECON>(d, wl, k, m, ta, tb, nc, UL, UR);
        double nh[3];
        shell_face_normal(shell_pts(d, e, nc), k, m, ta, tb, nh);
        PM pm;
        load_pm(d.metff + (int64_t)k * NPM * nfaces, nfaces, (int64_t)e * nfc + fi, pm);
        double nu[3];
        for (int i = 0; i < 3; ++i)
            nu[i] = fma(pm.gu[sym3(i, 0)], nh[0], fma(pm.gu[sym3(i, 1)], nh[1], pm.gu[sym3(i, 2)] * nh[2]));
        const double inrm = 1.0 / sqrt(d3(nu, nh));
        double nl[3];
        for (int i = 0; i < 3; ++i) nl[i] = nh[i] * inrm;
        const double lam = pm.a + fabs(d3(pm.b, nl));
        double hS[NQ], dU[NV], F[3][NV];
        for (int qq = 0; qq < NQ; ++qq) hS[qq] = 0.5 * (UL[qq] + UR[qq]);
        for (int v = 0; v < NV; ++v) dU[v] = UR[v] - UL[v];
        flux_gen(hS, hS + NV, pm, F);
        for (int j = 0; j < 3; ++j) {
            const double hn = -0.5 * lam * nu[j] * inrm;
            for (int v = 0; v < NV; ++v) flux_at_c(d, k, j, v, wl)[face_index(nc, m, ta, tb)] = fma(hn, dU[v], F[j][v]);
        }
    }
}

// One thread per (chunk position, cell): flux difference + sources + stage.
// KS: the Kerr-Schild background (metric and its derivative terms at the
// subcell centre from Dev::metfd; sources, stiff solve, clamp and implicit
// operator in their metric-general forms).  FACES: the flux components of every
// face instead of its states.
template <int SUB, bool CURVED, bool KS = false, bool FACES = KS>
__global__ void k_fd_update(Dev d, const int* list, int ci, int w0, SubArgs a) {
    const int n = chunk_n(d, ci, w0);
    const int64_t total = (int64_t)n * d.ncell;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        const int wl = (int)(q / d.ncell), c = (int)(q % d.ncell);
        const int e = list[w0 + wl];
        const ES es = esz(d, e);
        if (c >= es.ncell) continue;
        const int nc = es.nc;
        const int cc[3] = {c % nc, (c / nc) % nc, c / (nc * nc)};
        const int64_t p = fdb(d, e) + c;
        double ij[3][3];
        ShellPts sp;
        if (CURVED) {
            sp = shell_pts(d, e, nc);
            shell_cell(sp, cc, ij, nullptr);
        }
        double du[NV], u0[NV];
        for (int v = 0; v < NV; ++v) u0[v] = a.Uin.fd(v)[p];
        PM m;
        const int64_t mstride = (int64_t)d.E * d.ncell, mp = (int64_t)e * d.ncell + c;
        if (KS) {
            load_pm(d.metfd, mstride, mp, m);
            const double jd[3] = {a.J.fd(0)[p], a.J.fd(1)[p], a.J.fd(2)[p]};
            sources_gen(u0, jd, m, d.metfd, mstride, mp, du);
        } else {
            du[0] = -a.J.fd(0)[p];
            du[1] = -a.J.fd(1)[p];
            du[2] = -a.J.fd(2)[p];
            du[3] = du[4] = du[5] = 0.0;
            du[6] = u0[8];
            du[7] = du[8] = 0.0;
        }
        for (int k = 0; k < 3; ++k) {
            int t1, t2;
            axes_of(k, t1, t2);
            const int f0 = face_index(nc, cc[k], cc[t1], cc[t2]), f1 = f0 + nc * nc;
            if (FACES) {
                for (int j = 0; j < 3; ++j) {
                    const double sc = ij[k][j] * (0.5 * nc);
                    for (int v = 0; v < NV; ++v) {
                        const double* fl = flux_at_c(d, k, j, v, wl);
                        du[v] = fma(-sc, fl[f1] - fl[f0], du[v]);
                    }
                }
            } else if (CURVED) {
                // F^j = F^j(G) - n^_j D at each face (k_fd_states)
                double dG[NQ], sc[3];
                for (int q = 0; q < NQ; ++q) {
                    const double* g = fstate_at(d, k, q, wl);
                    dG[q] = g[f1] - g[f0];
                }
                for (int j = 0; j < 3; ++j) sc[j] = ij[k][j] * (0.5 * nc);
                flux_div_flat(dG, sc, du);
                const double s0 = (0.5 * nc) * shell_grad_normal(sp, k, cc, cc[k], ij[k]);
                const double s1 = (0.5 * nc) * shell_grad_normal(sp, k, cc, cc[k] + 1, ij[k]);
                for (int v = 0; v < NV; ++v) {
                    const double* g = fstate_at(d, k, NQ + v, wl);
                    du[v] = fma(s1, g[f1], fma(-s0, g[f0], du[v]));
                }
            } else {
                const double sc = d.ijac[3 * e + k] * (0.5 * nc);
                for (int v = 0; v < NV; ++v) {
                    const double* fl = flux_at(d, k, v, wl);
                    du[v] = fma(-sc, fl[f1] - fl[f0], du[v]);
                }
            }
        }
        if (SUB == SUB_RHS) {
            for (int v = 0; v < NV; ++v) a.Fout.fd(v)[p] = du[v];
            continue;
        }
        if (c == 0) {
            atomicAdd(d.units, (unsigned long long)es.ncell);
            atomicAdd(d.units + 1, 1ull);
        }
        if (SUB != SUB_C)
            for (int v = 0; v < NV; ++v) a.Fout.fd(v)[p] = du[v];
        double u[NV];
        substep_explicit(SUB, du, p, true, a, solve_k(d, e), u);
        if (KS) {
            if (SUB != SUB_C && !stiff_solve_gen(u, m, d, dt_of(d, e) * IM_A)) atomic_status(d, 2);
            if (d.mode != FFE_RELAX) hard_clamp_gen(u, m);
            if (SUB != SUB_C) {
                double g[NG];
                implicit_G_gen(u, m, d, g);
                for (int cg = 0; cg < NG; ++cg) a.Gout.fd(cg)[p] = g[cg];
            }
        } else {
            substep_implicit<SUB>(d, solve_k(d, e), a, p, true, u);
        }
        bool bad = false;
        for (int v = 0; v < NV; ++v) {
            a.Uout.fd(v)[p] = u[v];
            bad |= !is_finite(u[v]);
        }
        if (bad) atomic_status(d, 1);
    }
}

int fd_chunks(const Dev& d) { return (d.fd_cap + d.chunk - 1) / d.chunk; }

static size_t ghost_smem(const Dev& d) {
    return (size_t)(NQ * d.nn + NQ * GH * d.np1 * d.np1 + NQ * GH * d.nc * d.np1) * sizeof(double);
}

void launch_fd_fill(const Dev& d, const int* list, int ci, int w0, Field U, Field J, cudaStream_t st, bool residues,
                    bool traces) {
    const size_t smem = ghost_smem(d);
    cudaFuncSetAttribute(k_fd_fill, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_fd_fill<<<d.nsm * 4, 256, smem, st>>>(d, list, ci, w0, U, J, residues, traces);
    g_launch_counter += 1;
}

template <int SUB>
static void launch_update(const Dev& d, const int* list, int ci, int w0, const SubArgs& a, cudaStream_t st) {
    if (d.ks) k_fd_update<SUB, true, true><<<d.nsm * 8, 256, 0, st>>>(d, list, ci, w0, a);
    else if (d.curved) k_fd_update<SUB, true><<<d.nsm * 8, 256, 0, st>>>(d, list, ci, w0, a);
    else k_fd_update<SUB, false><<<d.nsm * 8, 256, 0, st>>>(d, list, ci, w0, a);
}

void launch_fd_substep(const Dev& d, int sub, const int* list, int ci, Field Uin, Field J, Field un, Field F2,
                       Field F3, Field G1, Field G2, Field G3, Field G4, Field Fout, Field Uout, Field Gout,
                       Field Jout, cudaStream_t st, bool faces) {
    SubArgs a{Uin, J, un, F2, F3, G1, G2, G3, G4, Fout, Uout, Gout, Jout};
    const int grid = d.nsm * 8;
    for (int k = 0, nch = fd_chunks(d); k < nch; ++k) {
        const int w0 = k * d.chunk;
        prof_begin("fd_fill", st);
        launch_fd_fill(d, list, ci, w0, Uin, J, st, faces, ci == 1);
        prof_end(st);
        prof_begin("fd_flux", st);
        if (faces) {
            k_fd_flux_faces<<<grid, 128, 0, st>>>(d, list, ci, w0);
        } else if (d.recon == FFE_RECON_MP5) {
            if (d.ks) k_fd_flux_ks<FFE_RECON_MP5><<<grid, 128, 0, st>>>(d, list, ci, w0);
            else if (d.curved) k_fd_states<FFE_RECON_MP5><<<grid, 64, 0, st>>>(d, list, ci, w0);
            else k_fd_flux<FFE_RECON_MP5><<<grid, 64, 0, st>>>(d, list, ci, w0);
        } else {
            if (d.ks) k_fd_flux_ks<FFE_RECON_WENO5Z><<<grid, 128, 0, st>>>(d, list, ci, w0);
            else if (d.curved) k_fd_states<FFE_RECON_WENO5Z><<<grid, 64, 0, st>>>(d, list, ci, w0);
            else k_fd_flux<FFE_RECON_WENO5Z><<<grid, 64, 0, st>>>(d, list, ci, w0);
        }
        prof_end(st);
        prof_begin("fd_update", st);
        switch (sub) {
            case SUB_A: launch_update<SUB_A>(d, list, ci, w0, a, st); break;
            case SUB_B: launch_update<SUB_B>(d, list, ci, w0, a, st); break;
            case SUB_C: launch_update<SUB_C>(d, list, ci, w0, a, st); break;
            default:
                if (faces) k_fd_update<SUB_RHS, true, false, true><<<d.nsm * 8, 256, 0, st>>>(d, list, ci, w0, a);
                else launch_update<SUB_RHS>(d, list, ci, w0, a, st);
        }
        prof_end(st);
        g_launch_counter += 2;
    }
}

// ---------------------------------------------------------------------------
// DG -> FD projection (tensor Lagrange evaluation at subcell centres) of `nv`
// variables of element e, from its DG slot to its FD slot, all at once.
__device__ void project_dg2fd_element(const Dev& d, const Field& F, int nv, int e, double* sm) {
    const ES es = esz(d, e);
    const Tables& T = d.tabs[es.P];
    const int np1 = es.np1, nc = es.nc, nb = nc * np1 * np1, ncc = nc * nc * np1;
    const int64_t fb = fdb(d, e);
    double* b = sm;                 // [nv][np1][np1][nc]
    double* c = b + nv * nb;        // [nv][np1][nc][nc]
    for (int t = threadIdx.x; t < nv * nb; t += blockDim.x) {
        const int v = t / nb, x = t % nc, jk = (t % nb) / nc;
        const double* src = F.dg(v) + (int64_t)e * d.nn + np1 * jk;
        double acc = 0.0;
        for (int m = 0; m < np1; ++m) acc = fma(T.P2F[x][m], src[m], acc);
        b[t] = acc;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nv * ncc; t += blockDim.x) {
        const int v = t / ncc, r = t % ncc, x = r % nc, y = (r / nc) % nc, k = r / (nc * nc);
        double acc = 0.0;
        for (int m = 0; m < np1; ++m) acc = fma(T.P2F[y][m], b[v * nb + x + nc * (m + np1 * k)], acc);
        c[t] = acc;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nv * es.ncell; t += blockDim.x) {
        const int v = t / es.ncell, r = t % es.ncell, xy = r % (nc * nc), z = r / (nc * nc);
        double acc = 0.0;
        for (int m = 0; m < np1; ++m) acc = fma(T.P2F[z][m], c[v * ncc + xy + nc * nc * m], acc);
        F.fd(v)[fb + r] = acc;
    }
    __syncthreads();
}

struct RollArgs {
    Field f[8];
    int nv[8];
    int nf;
    Field J;   // J~ of the stage state (f[1])
};

// Flagged elements (the indicator gave each an FD slot): one CTA per (element,
// field) projects a substep input to the subcells; the one of the stage state also
// forms J~ there and marks the element FD.
__global__ void k_rollback_project(Dev d, RollArgs r) {
    extern __shared__ double sm[];
    const int n = d.counts[2];
    for (int w = blockIdx.x; w < n * r.nf; w += gridDim.x) {
        const int e = d.flag_list[w / r.nf], i = w % r.nf;
        project_dg2fd_element(d, r.f[i], r.nv[i], e, sm);
        if (i == 1) {
            if (threadIdx.x == 0) d.mask[e] = 1;
            __syncthreads();
            for (int c = threadIdx.x; c < d.ncell; c += blockDim.x) current_fd_cell(d, e, c, r.f[1], r.J);
        }
    }
}

void launch_rollback_project(const Dev& d, int sub, Field un, Field Uin, Field J, Field F2, Field F3, Field G1, Field G2,
                             Field G3, Field G4, cudaStream_t st) {
    RollArgs r{};
    r.J = J;
    int k = 0;
    auto add = [&](Field f, int nv) {
        r.f[k] = f;
        r.nv[k] = nv;
        ++k;
    };
    add(un, NV);
    add(Uin, NV);
    if (sub == SUB_A) { add(G1, NG); add(G2, NG); }
    if (sub == SUB_B) { add(F2, NV); add(G1, NG); add(G2, NG); add(G3, NG); }
    if (sub == SUB_C) { add(F2, NV); add(F3, NV); add(G2, NG); add(G3, NG); add(G4, NG); }
    r.nf = k;
    const int np1 = d.np1, nc = d.nc;
    const size_t smem = (size_t)NV * (nc * np1 * np1 + nc * nc * np1) * sizeof(double);
    cudaFuncSetAttribute(k_rollback_project, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    prof_begin("rollback_project", st);
    k_rollback_project<<<d.nsm * 2, 256, smem, st>>>(d, r);
    prof_end(st);
    g_launch_counter += 1;
}

// ---------------------------------------------------------------------------
// FD -> DG (6-point Lagrange per direction) of nv variable blocks ([nc^3], one
// every `stride` doubles from src) into dst ([nv][np1^3]), sum-factorised through
// shared memory, all variables at once.
__device__ void project_fd2dg_vars(const ES& es, const Tables& T, const double* src, int64_t stride, int nv, double* dst,
                                   double* sm) {
    const int np1 = es.np1, nc = es.nc, nb = nc * nc * np1, ncc = nc * np1 * np1, nn = es.nn;
    double* b = sm;                // [nv][nc][nc][np1]
    double* c = b + nv * nb;       // [nv][nc][np1][np1]
    for (int t = threadIdx.x; t < nv * nb; t += blockDim.x) {
        const int v = t / nb, i = t % np1, yz = (t % nb) / np1;
        const int lo = T.f2d_lo[i];
        const double* a = src + v * stride + lo + nc * yz;
        double acc = 0.0;
        for (int m = 0; m < 6; ++m) acc = fma(T.F2D[i][lo + m], a[m], acc);
        b[t] = acc;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nv * ncc; t += blockDim.x) {
        const int v = t / ncc, r = t % ncc, i = r % np1, j = (r / np1) % np1, z = r / (np1 * np1);
        const int lo = T.f2d_lo[j];
        double acc = 0.0;
        for (int m = 0; m < 6; ++m) acc = fma(T.F2D[j][lo + m], b[v * nb + i + np1 * ((lo + m) + nc * z)], acc);
        c[t] = acc;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nv * nn; t += blockDim.x) {
        const int v = t / nn, r = t % nn, ij = r % (np1 * np1), k = r / (np1 * np1);
        const int lo = T.f2d_lo[k];
        double acc = 0.0;
        for (int m = 0; m < 6; ++m) acc = fma(T.F2D[k][lo + m], c[v * ncc + ij + np1 * np1 * (lo + m)], acc);
        dst[t] = acc;
    }
    __syncthreads();
}

// shared doubles of k_fd2dg: projection scratch of 6 variables | B~ [3][nn] or 6 variables
// [6][nn] | tmp [3][nn] | red [2][8]
static size_t fd2dg_smem(const Dev& d) {
    return (size_t)(6 * (d.nc * d.nc * d.np1 + d.nc * d.np1 * d.np1) + 9 * d.nn + 16) * sizeof(double);
}

// End of step: FD elements that did not switch during the step return to DG
// when the indicator with alpha' = alpha + 1 finds their FD->DG projection
// admissible; their FD slot returns to the pool.
__global__ void __launch_bounds__(256) k_fd2dg(Dev d, Field un) {
    extern __shared__ double sm[];
    const int n = d.counts[1];
    for (int w = blockIdx.x; w < n; w += gridDim.x) {
        const int e = d.fd_list[w];
        if (d.switched[e]) continue;
        const ES es = esz(d, e);
        const Tables& T = d.tabs[es.P];
        const int np1 = es.np1, nn = es.nn;
        double* work = sm;                                                     // projection scratch
        double* proj = work + 6 * (d.nc * d.nc * d.np1 + d.nc * d.np1 * d.np1);   // [6][nn]
        double* tmp = proj + 6 * d.nn;                                         // [3][nn]
        double* red = tmp + 3 * d.nn;                                          // [2][8]
        const int64_t fb = fdb(d, e), db = (int64_t)e * d.nn;
        project_fd2dg_vars(es, T, un.fd(3) + fb, un.nfd, 3, proj, work);
        for (int t = threadIdx.x; t < nn; t += blockDim.x) {
            const double bx = proj[t], by = proj[nn + t], bz = proj[2 * nn + t];
            if (d.ks) {
                // |B~| with the spatial metric at the node
                PM m;
                load_pm(d.met, d.ndg, db + t, m);
                const double u[NV] = {0.0, 0.0, 0.0, bx, by, bz, 0.0, 0.0, 0.0};
                tmp[t] = bnorm_gen(u, m);
            } else {
                tmp[t] = sqrt(fma(bz, bz, fma(by, by, bx * bx)));
            }
        }
        __syncthreads();
        for (int t = threadIdx.x; t < nn; t += blockDim.x) {
            const int i = t % np1, j = (t / np1) % np1, k = t / (np1 * np1);
            double acc = 0.0;
            for (int m = 0; m < np1; ++m) acc = fma(T.Pi[i][m], tmp[m + np1 * (j + np1 * k)], acc);
            tmp[nn + t] = acc;
        }
        __syncthreads();
        for (int t = threadIdx.x; t < nn; t += blockDim.x) {
            const int i = t % np1, j = (t / np1) % np1, k = t / (np1 * np1);
            double acc = 0.0;
            for (int m = 0; m < np1; ++m) acc = fma(T.Pi[j][m], tmp[nn + i + np1 * (m + np1 * k)], acc);
            tmp[2 * nn + t] = acc;
        }
        __syncthreads();
        // third low-pass direction and the two sums: per-thread partial sums in a fixed
        // order, then a fixed tree over the lanes and the warps (deterministic)
        double pn = 0.0, pd = 0.0;
        for (int t = threadIdx.x; t < nn; t += blockDim.x) {
            const int i = t % np1, j = (t / np1) % np1;
            double acc = 0.0;
            for (int m = 0; m < np1; ++m) acc = fma(T.Pi[t / (np1 * np1)][m], tmp[2 * nn + i + np1 * (j + np1 * m)], acc);
            const double uh = tmp[t] - acc;
            pn = fma(uh, uh, pn);
            pd = fma(tmp[t], tmp[t], pd);
        }
        for (int o = 16; o > 0; o >>= 1) {
            pn += __shfl_down_sync(0xffffffffu, pn, o);
            pd += __shfl_down_sync(0xffffffffu, pd, o);
        }
        if ((threadIdx.x & 31) == 0) {
            red[threadIdx.x >> 5] = pn;
            red[8 + (threadIdx.x >> 5)] = pd;
        }
        __syncthreads();
        double num = 0.0, den = 0.0;
        for (int i = 0; i < (int)blockDim.x / 32; ++i) { num += red[i]; den += red[8 + i]; }
        const double thr = d.thr_fdP[es.P];
        const double ratio = den > 0.0 ? sqrt(num / den) : 0.0;
        if (threadIdx.x == 0 && fabs(ratio - thr) <= 1e-12 * thr) d.near_list[atomicAdd(&d.counts[3], 1) & 4095] = e;
        if (!(ratio > thr)) {
            for (int t = threadIdx.x; t < 3 * nn; t += blockDim.x) un.dg(3 + t / nn)[db + t % nn] = proj[t];
            __syncthreads();
            project_fd2dg_vars(es, T, un.fd(0) + fb, un.nfd, 3, proj, work);
            project_fd2dg_vars(es, T, un.fd(6) + fb, un.nfd, 3, proj + 3 * nn, work);
            for (int t = threadIdx.x; t < 6 * nn; t += blockDim.x) {
                const int v = t / nn;
                un.dg(v < 3 ? v : v + 3)[db + t % nn] = proj[t];
            }
            if (threadIdx.x == 0) {
                d.mask[e] = 0;
                if (d.fd_slot) {
                    const int sl = d.fd_slot[e];
                    d.fd_slot[e] = -1;
                    d.slot_elem[sl] = -1;
                    d.free_slots[atomicAdd(&d.counts[5], 1)] = sl;
                }
            }
        }
        __syncthreads();
    }
}

void launch_fd2dg(const Dev& d, Field un, cudaStream_t st) {
    const size_t smem = fd2dg_smem(d);
    cudaFuncSetAttribute(k_fd2dg, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    prof_begin("fd2dg", st);
    k_fd2dg<<<d.nsm * 2, 256, smem, st>>>(d, un);
    prof_end(st);
    g_launch_counter += 1;
}

// ---------------------------------------------------------------------------
// The WENO5-Z reciprocal, elementwise (accuracy tests of recip_nr).
__global__ void k_eval_recip(const double* x, double* y, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = recip_nr(x[i]);
}

void launch_eval_recip(const double* x, double* y, int64_t n, cudaStream_t st) {
    const int64_t blocks = (n + 255) / 256;
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        nsm < 1)
        nsm = 1;
    const int cap = nsm * 16;
    k_eval_recip<<<(int)(blocks < cap ? blocks : cap), 256, 0, st>>>(x, y, n);
    g_launch_counter += 1;
}

// ---------------------------------------------------------------------------
// FP64 FMA throughput probe (the measured denominator of the FP64 roofline):
// every thread runs 8 independent DFMA chains in registers, no memory traffic;
// the chains stay live through a store that the data never trigger.
__device__ double g_fma_sink;

__global__ void k_fma_probe(int iters, double a, double b) {
    double x[8];
    for (int k = 0; k < 8; ++k) x[k] = threadIdx.x * 1e-3 + k;
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = fma(x[k], a, b);
    }
    double acc = 0.0;
    for (int k = 0; k < 8; ++k) acc += x[k];
    if (acc == -1.0) g_fma_sink = acc;
}

double launch_fma_probe(int nsm, int iters, cudaStream_t st, float* ms) {
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    const int blocks = nsm * 4, threads = 256;
    k_fma_probe<<<blocks, threads, 0, st>>>(iters / 8 + 1, 0.999999, 1e-7);   // warm-up
    cudaEventRecord(e0, st);
    k_fma_probe<<<blocks, threads, 0, st>>>(iters, 0.999999, 1e-7);
    cudaEventRecord(e1, st);
    cudaEventSynchronize(e1);
    cudaEventElapsedTime(ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    g_launch_counter += 2;
    return 2.0 * 8.0 * (double)iters * blocks * threads;
}

}  // namespace ffe
