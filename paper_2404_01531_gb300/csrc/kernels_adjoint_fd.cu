// Reverse mode of the FD-subcell right-hand side on flat-metric shells
// (Sec. III.C.2), for a fixed DG/FD mask:
//   out += (d RHS_FD / d U)^T lambda  over every listed FD element.
// The forward operator of an FD element is: extended block of the 12
// quantities (U and J~ = J~(U)) with 3 ghost layers from FD neighbours
// (copies; interpolated along the edge across faces between wedges), DG neighbours (their polynomials of U and of the nodal J~ at the
// ghost subcell centres) or the boundary states; WENO5-Z left/right values at every face; Rusanov flux
// of every physical component with the unit face normal; optional 4th-order
// corrector with the cell-centred fluxes; flux difference with the inverse
// Jacobian at the cell centre; sources -J~_drift and q~.
//   k_fdv_lines   face-state adjoints from the two cells' lambda (k_fdv_cell_weights),
//                 back through corrector, Rusanov and WENO5-Z along every line;
//                 k_fdv_gather sums the lines into the extended-block adjoint
//   k_fdv_cells   interior positions of the extended-block adjoint (U and the
//                 current's chain rule) and the source terms, into out
//   k_fdv_ghosts  ghost positions: into the FD neighbour's cells, through the
//                 transposed DG -> FD evaluation (of U and of the nodal J~) into
//                 the DG neighbour's nodes, or through the boundary state into my
//                 outermost cells
// The lines' contributions to the extended-block adjoint are summed per cell in
// a fixed order (k_fdv_gather); where
// several elements meet in out (an element's cells, a neighbour's cells or
// nodes reached through ghosts) they are summed with FP64 atomics (the order
// of those additions, hence the last bits, may differ between runs).
#include "ffe_internal.h"
#include "physics.cuh"
#include "shellmap.cuh"
#include "fd_common.cuh"
#include "adjoint_common.cuh"

namespace ffe {

__device__ __forceinline__ double* extb_at(const Dev& d, double* extb, int q, int wl) {
    return extb + ((int64_t)q * d.chunk + wl) * ext_size(d);
}


// Scratch of the FD reverse mode, per chunk position (gb):
//   H [3][12][nc^3]   per cell and direction k, the adjoint of the face states' G it
//                     owes: F^j = F^j(G) - n^_j D (k_fd_states) enters the cell as
//                     du -= (nc/2) d_j xi^k (F^j(right) - F^j(left)), so G of its right
//                     face receives -H and G of its left face +H, H_q = -dF^j/dG_q summed
//   S [3][2][nc^3]    (nc/2) grad xi^k . n^ at its left and right face (D's factor)
//   V [3][12][nc^2 (nc+6)]  the adjoint of every cell of every line, ghosts included
__device__ __forceinline__ int64_t vline(const Dev& d) { return (int64_t)d.nc * d.nc * (d.nc + 2 * GH); }
__device__ __forceinline__ double* h_at(const Dev& d, double* gb, int k, int q, int wl) {
    return gb + (((int64_t)k * NQ + q) * d.chunk + wl) * d.ncell;
}
__device__ __forceinline__ double* s_at(const Dev& d, double* gb, int k, int side, int wl) {
    return gb + (int64_t)3 * NQ * d.chunk * d.ncell + (((int64_t)k * 2 + side) * d.chunk + wl) * d.ncell;
}
__device__ __forceinline__ double* v_at(const Dev& d, double* gb, int k, int q, int wl) {
    return gb + (int64_t)(3 * NQ + 6) * d.chunk * d.ncell + (((int64_t)k * NQ + q) * d.chunk + wl) * vline(d);
}
size_t fdv_scratch(const Dev& d, int chunk) {
    const size_t nc = d.nc;
    return ((size_t)(3 * NQ + 6) * d.ncell + (size_t)3 * NQ * nc * nc * (nc + 2 * GH)) * chunk;
}

__global__ void k_fdv_cell_weights(Dev d, const int* list, int ci, int w0, Field L, double* gb) {
    const int n = chunk_n(d, ci, w0);
    const int64_t total = (int64_t)n * d.ncell;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int wl = (int)(t / d.ncell), c = (int)(t % d.ncell);
        const int e = list[w0 + wl];
        const ES es = esz(d, e);
        if (c >= es.ncell) continue;
        const int nc = es.nc;
        const int cc[3] = {c % nc, (c / nc) % nc, c / (nc * nc)};
        const ShellPts sp = shell_pts(d, e, nc);
        double ij[3][3], l[NV];
        shell_cell(sp, cc, ij, nullptr);
        for (int v = 0; v < NV; ++v) l[v] = L.fd(v)[fdb(d, e) + c];
        for (int k = 0; k < 3; ++k) {
            const double a = ij[k][0] * (0.5 * nc), b = ij[k][1] * (0.5 * nc), g = ij[k][2] * (0.5 * nc);
            // transpose of flux_div_flat
            h_at(d, gb, k, 0, wl)[c] = fma(-g, l[4], fma(b, l[5], -a * l[6]));
            h_at(d, gb, k, 1, wl)[c] = fma(g, l[3], fma(-a, l[5], -b * l[6]));
            h_at(d, gb, k, 2, wl)[c] = fma(-b, l[3], fma(a, l[4], -g * l[6]));
            h_at(d, gb, k, 3, wl)[c] = fma(g, l[1], fma(-b, l[2], -a * l[7]));
            h_at(d, gb, k, 4, wl)[c] = fma(-g, l[0], fma(a, l[2], -b * l[7]));
            h_at(d, gb, k, 5, wl)[c] = fma(b, l[0], fma(-a, l[1], -g * l[7]));
            h_at(d, gb, k, 6, wl)[c] = -fma(a, l[0], fma(b, l[1], g * l[2]));
            h_at(d, gb, k, 7, wl)[c] = -fma(a, l[3], fma(b, l[4], g * l[5]));
            h_at(d, gb, k, 8, wl)[c] = 0.0;
            h_at(d, gb, k, 9, wl)[c] = -a * l[8];
            h_at(d, gb, k, 10, wl)[c] = -b * l[8];
            h_at(d, gb, k, 11, wl)[c] = -g * l[8];
            for (int side = 0; side < 2; ++side)
                s_at(d, gb, k, side, wl)[c] = (0.5 * nc) * shell_grad_normal(sp, k, cc, cc[k] + side, ij[k]);
        }
    }
}

// One thread per (chunk position, direction, quantity, line): marches the line as
// the forward kernel does (Weno5zLine), with the adjoints of the window's
// differences in registers, and writes each cell's adjoint once it is complete.
// The indicators and Z weights of a cell are formed once for its two face
// values, where a thread per face forms them, and their reverse, twice; no
// per-face contributions go through memory: 54 elements 1.36 -> 0.90 ms, 0.84 with
// the candidates by their differences from the central one.
__global__ void __launch_bounds__(64, 8) k_fdv_lines(Dev d, const int* list, int ci, int w0, Field L, double* gb) {
    const int n = chunk_n(d, ci, w0);
    const int nlm = d.nc * d.nc, per = 3 * NQ * nlm;
    const int64_t total = (int64_t)n * per;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int wl = (int)(t / per), r = (int)(t % per), line = r % nlm, kq = r / nlm;
        const int k = kq / NQ, q = kq % NQ;
        const int e = list[w0 + wl];
        const int nc = esz(d, e).nc, nl = nc * nc;
        if (line >= nl) continue;
        const int ta = line % nc, tb = line / nc;
        int64_t stride;
        const double* pv = ext_at(d, q, wl) + line_start(k, ta, tb, nc, stride);
        // the line's cells inside the element
        const int cs[3] = {1, nc, nc * nc};
        int t1, t2;
        axes_of(k, t1, t2);
        const int c0 = ta * cs[t1] + tb * cs[t2], step = cs[k];
        const double* ph = h_at(d, gb, k, q, wl) + c0;
        const double* p0 = s_at(d, gb, k, 0, wl) + c0;
        const double* p1 = s_at(d, gb, k, 1, wl) + c0;
        const double* pl = q < NV ? L.fd(q) + fdb(d, e) + c0 : nullptr;
        const bool corr = d.fd_corr;
        const double c1 = corr ? 2.0 / 3.0 : 0.5;
        // adjoints of the face m's left and right state and of the sum of its two cells
        auto face = [&](int m, double& lb, double& rb) {
            double G = 0.0, D = 0.0;
            if (m > 0) {
                G = ph[(m - 1) * step];
                if (pl) D = p1[(m - 1) * step] * pl[(m - 1) * step];
            }
            if (m < nc) {
                G -= ph[m * step];
                if (pl) D = fma(-p0[m * step], pl[m * step], D);
            }
            lb = c1 * (G - D);
            rb = c1 * (G + D);
            return corr ? (-1.0 / 6.0) * G : 0.0;
        };
        Weno5zLineVjp A;
        A.init(pv[0], pv[stride], pv[2 * stride], pv[3 * stride], d.weno_eps);
        double* out = v_at(d, gb, k, q, wl) + line;
        // window at centre c (extended index): hb0..2 at c-1..c+1, differences
        // (c-2,c-1) .. (c,c+1) in g0, g1, g2; cells c-2 .. c+1 not yet written hold their
        // direct adjoints in v0 (c-2) .. v3 (c+1)
        double hb0 = 0.0, hb1 = 0.0, hb2, g0 = 0.0, g1 = 0.0, g2, gm = 0.0;
        double L0, R0, S0 = face(0, L0, R0);
        double va = 0.0, vb = 0.0, vc = S0, vd;   // direct adjoints of cells c-2, c-1, c, c+1
#pragma unroll 1
        for (int c = GH - 1; c <= nc + GH; ++c) {
            // centre c: right value -> left state of face c-2, left value -> right state of face c-3
            const bool left = c > GH - 1, right = c < nc + GH;
            double yl = 0.0, yr = 0.0;
            vd = 0.0;
            if (left) {
                yl = R0;       // of face c-3, read one cell ago
                if (right) {
                    S0 = face(c - 2, L0, R0);
                    yr = L0;
                    vc += S0;
                    vd = S0;
                }
            } else {
                yr = L0;
                vd = S0;
            }
            hb2 = 0.0;
            g2 = 0.0;
            A.cell(pv[(c + 2) * stride], yl, yr, hb0, hb1, hb2, g1, g2);
            vc += yl + yr;
            // h at c-1 is complete: h = (d(c-1,c) - d(c-2,c-1))/8
            const double h8 = 0.125 * hb0;
            g1 += h8;
            g0 -= h8;
            // d(c-2,c-1) is complete, and with it cell c-2 (gm: d(c-3,c-2))
            out[(c - 2) * nl] = va + (gm - g0);
            gm = g0; g0 = g1; g1 = g2;
            hb0 = hb1; hb1 = hb2;
            va = vb; vb = vc; vc = vd;
        }
        // after the last centre c = nc + GH: the window stands at c + 1 = nc + GH + 1
        {
            const int c = nc + GH + 1;
            // h at c-1 and c hold what the last centres left
            double h8 = 0.125 * hb0;
            g1 += h8;
            g0 -= h8;
            out[(c - 2) * nl] = va + (gm - g0);
            gm = g0; g0 = g1; g1 = 0.0;
            h8 = 0.125 * hb1;
            g1 += h8;
            g0 -= h8;
            out[(c - 1) * nl] = vb + (gm - g0);
            gm = g0; g0 = g1;
            out[c * nl] = vc + (gm - g0);
            out[(c + 1) * nl] = g0;
        }
    }
}

// Extended-block adjoint of cell (x, y, z) and quantity q: the sum of the lines of
// the three directions that hold it; every position is written, no clearing, no
// atomics, a fixed order.
__global__ void k_fdv_gather(Dev d, const int* list, int ci, int w0, double* gb, double* extb) {
    const int n = chunk_n(d, ci, w0);
    const int64_t ext = ext_size(d);
    const int64_t total = (int64_t)n * NQ * ext;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int wl = (int)(t / (NQ * ext));
        const int qq = (int)((t / ext) % NQ);
        const int o = (int)(t % ext);
        const int e = list[w0 + wl];
        const int nc = esz(d, e).nc, ne = nc + 2 * GH;
        if (o >= ne * ne * ne) continue;
        const int c3[3] = {o % ne, (o / ne) % ne, o / (ne * ne)};
        double acc = 0.0;
        for (int k = 0; k < 3; ++k) {
            int t1, t2;
            axes_of(k, t1, t2);
            const int ta = c3[t1] - GH, tb = c3[t2] - GH;
            if (ta < 0 || ta >= nc || tb < 0 || tb >= nc) continue;
            acc += v_at(d, gb, k, qq, wl)[ta + nc * (tb + nc * c3[k])];
        }
        extb_at(d, extb, qq, wl)[o] = acc;
    }
}

__global__ void k_fdv_cells(Dev d, const int* list, int ci, int w0, Field U, Field L, Field out, const double* extb) {
    const int n = chunk_n(d, ci, w0);
    const int64_t total = (int64_t)n * d.ncell;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        const int wl = (int)(q / d.ncell), c = (int)(q % d.ncell);
        const int e = list[w0 + wl];
        const ES es = esz(d, e);
        if (c >= es.ncell) continue;
        const int nc = es.nc, ne = nc + 2 * GH;
        const int x = c % nc, y = (c / nc) % nc, z = c / (nc * nc);
        const int64_t o = (x + GH) + ne * ((y + GH) + ne * (z + GH));
        const int64_t p = fdb(d, e) + c;
        double u[NV], ub[NV], jb[3];
        for (int v = 0; v < NV; ++v) {
            u[v] = U.fd(v)[p];
            ub[v] = extb_at(d, (double*)extb, v, wl)[o];
        }
        for (int k = 0; k < 3; ++k) jb[k] = extb_at(d, (double*)extb, NV + k, wl)[o];
        current_vjp(u, d.eta, jb, jb, ub);   // the extended block holds J~ = J~(U)
        const double wd[3] = {-L.fd(0)[p], -L.fd(1)[p], -L.fd(2)[p]}, zero[3] = {0.0, 0.0, 0.0};
        current_vjp(u, d.eta, wd, zero, ub);  // source -J~_drift
        ub[8] += L.fd(6)[p];                  // source q~ in the psi~ equation
        for (int v = 0; v < NV; ++v)
            if (ub[v] != 0.0) atomicAdd(out.fd(v) + p, ub[v]);
    }
}

// shared doubles of one face's ghosts (U and J~): DG neighbour t1 [12][GH][np1][np1]
// | t2 [12][GH][np1][nc] | ub [12][GH][nc][nc]; FD neighbour across wedges
// W [GH][nc (its cell)][nc (ghost)] | ub [12][GH][nc][nc] (fits in the same)
size_t fdv_ghost_smem(const Dev& d) {
    return (size_t)(NQ * GH * d.np1 * d.np1 + NQ * GH * d.np1 * d.nc + NQ * GH * d.nc * d.nc) * sizeof(double);
}

__global__ void k_fdv_ghosts(Dev d, const int* list, int ci, int w0, Field U, Field J, Field out,
                             const double* extb, double* omega_bar) {
    const int n = chunk_n(d, ci, w0);
    extern __shared__ double sm[];
    __shared__ double s_om[256];
    double om_acc = 0.0;
    for (int item = blockIdx.x; item < n * 6; item += gridDim.x) {
        const int wl = item / 6, f = item % 6;
        const int e = list[w0 + wl];
        const int gsl = d.gislot ? d.gislot[e * 6 + f] : -1;   // a face between wedges: its weights (k_fd_fill)
        const ES es = esz(d, e);
        const Tables& T = d.tabs[es.P];
        const int nc = es.nc, ne = nc + 2 * GH, np1 = es.np1, nn = es.nn;
        const int dd = f >> 1, s = f & 1;
        int t1, t2;
        axes_of(dd, t1, t2);
        const int nb = d.nbr[e * 6 + f];
        const int nper = GH * nc * nc;
        auto ghost_offset = [&](int g, int ta, int tb) -> int64_t {
            int c[3];
            c[dd] = s ? nc + GH + g : GH - 1 - g;
            c[t1] = ta + GH;
            c[t2] = tb + GH;
            return c[0] + (int64_t)ne * (c[1] + (int64_t)ne * c[2]);
        };
        auto ghost_bar = [&](int64_t og, const double* u, double* ub) {
            double jb[3];
            for (int v = 0; v < NV; ++v) ub[v] = extb_at(d, (double*)extb, v, wl)[og];
            for (int k = 0; k < 3; ++k) jb[k] = extb_at(d, (double*)extb, NV + k, wl)[og];
            current_vjp(u, d.eta, jb, jb, ub);
        };
        if (nb >= 0 && d.mask[nb] == 1) {
            const int f2 = d.nbr_face[e * 6 + f];
            const int d2 = f2 >> 1, s2 = f2 & 1;
            int u1, u2;
            axes_of(d2, u1, u2);
            const int o = d.orient[e * 6 + f];
            const int64_t nbase = fdb(d, nb);
            if (gsl >= 0) {
                // Each cell (g, a2, radial tb) of the neighbour gathers its share of the
                // ghosts of its layer and radius through the transposed 6-point weights
                // along the edge (a small dense matrix in shared memory), then takes the
                // current's chain rule: one addition per cell and variable into out
                double* W = sm;
                double* ubo = W + GH * nc * nc;   // [12][GH][nc (tb)][nc (ta)]
                for (int t = threadIdx.x; t < GH * nc * nc; t += blockDim.x) {
                    const int g = t / (nc * nc), cell = (t / nc) % nc, ta = t % nc;
                    const int gi = gsl * GH * d.nc + g * nc + ta, m = cell - d.gst[gi];
                    W[t] = m >= 0 && m < 6 ? d.gwf[6 * (int64_t)gi + m] : 0.0;
                }
                for (int t = threadIdx.x; t < nper; t += blockDim.x) {
                    const int64_t og = ghost_offset(t / (nc * nc), t % nc, (t / nc) % nc);
                    for (int v = 0; v < NQ; ++v) ubo[v * nper + t] = extb_at(d, (double*)extb, v, wl)[og];
                }
                __syncthreads();
                for (int t = threadIdx.x; t < nper; t += blockDim.x) {
                    const int g = t / (nc * nc), cell = t % nc, tb = (t / nc) % nc;
                    int a2, b2;
                    orient_map(o, nc, 0, tb, a2, b2);
                    int c[3];
                    c[d2] = s2 ? nc - 1 - g : g;
                    c[u1] = cell;
                    c[u2] = b2;
                    const int64_t p = nbase + c[0] + nc * (c[1] + nc * c[2]);
                    double w[NQ];
                    for (int v = 0; v < NQ; ++v) w[v] = 0.0;
                    for (int ta = 0; ta < nc; ++ta) {
                        const double wt = W[(g * nc + cell) * nc + ta];
                        if (wt == 0.0) continue;
                        for (int v = 0; v < NQ; ++v) w[v] = fma(wt, ubo[v * nper + (g * nc + tb) * nc + ta], w[v]);
                    }
                    double u[NV];
                    for (int v = 0; v < NV; ++v) u[v] = U.fd(v)[p];
                    current_vjp(u, d.eta, w + NV, w + NV, w);
                    for (int v = 0; v < NV; ++v)
                        if (w[v] != 0.0) atomicAdd(out.fd(v) + p, w[v]);
                }
                __syncthreads();
                continue;
            }
            for (int t = threadIdx.x; t < nper; t += blockDim.x) {
                const int g = t / (nc * nc), ta = t % nc, tb = (t / nc) % nc;
                int a2, b2;
                orient_map(o, nc, ta, tb, a2, b2);
                int c[3];
                c[d2] = s2 ? nc - 1 - g : g;
                c[u1] = a2;
                c[u2] = b2;
                const int64_t p = nbase + c[0] + nc * (c[1] + nc * c[2]);
                double u[NV], ub[NV];
                for (int v = 0; v < NV; ++v) u[v] = U.fd(v)[p];
                ghost_bar(ghost_offset(g, ta, tb), u, ub);
                for (int v = 0; v < NV; ++v)
                    if (ub[v] != 0.0) atomicAdd(out.fd(v) + p, ub[v]);
            }
        } else if (nb >= 0) {
            const int f2 = d.nbr_face[e * 6 + f];
            const int d2 = f2 >> 1, s2 = f2 & 1;
            int u1, u2;
            axes_of(d2, u1, u2);
            const int o = d.orient[e * 6 + f];
            double* t1b = sm;                          // [12][GH][np1][np1]
            double* t2b = t1b + NQ * GH * np1 * np1;   // [12][GH][np1][nc]
            double* ubo = t2b + NQ * GH * np1 * nc;    // [12][GH][nc (u2)][nc (u1)]
            // The ghosts hold the neighbour's polynomial of U and of its nodal J~ at
            // its subcell centres: linear in (U, J~) at its nodes.  Their adjoints go
            // back through the transposed evaluation, then through J~(U) at each node.
            for (int t = threadIdx.x; t < nper; t += blockDim.x) {
                const int g = t / (nc * nc), ta = t % nc, tb = (t / nc) % nc;
                int a2, b2;   // the neighbour's subcell (along u1, u2) under this ghost cell
                orient_map(o, nc, ta, tb, a2, b2);
                if (gsl >= 0) a2 = ta;
                const int64_t og = ghost_offset(g, ta, tb);
                for (int v = 0; v < NQ; ++v)
                    ubo[((v * GH + g) * nc + b2) * nc + a2] = extb_at(d, (double*)extb, v, wl)[og];
            }
            __syncthreads();
            // ub -> t2-bar [v][g][m (u2 node)][a2 (u1 cell)]
            for (int t = threadIdx.x; t < NQ * GH * np1 * nc; t += blockDim.x) {
                const int v = t / (GH * np1 * nc), r = t % (GH * np1 * nc);
                const int g = r / (np1 * nc), mm = (r / nc) % np1, a2 = r % nc;
                double acc = 0.0;
                for (int b2 = 0; b2 < nc; ++b2) acc = fma(T.P2F[b2][mm], ubo[((v * GH + g) * nc + b2) * nc + a2], acc);
                t2b[((v * GH + g) * np1 + mm) * nc + a2] = acc;
            }
            __syncthreads();
            // t2-bar -> t1-bar [v][g][a2 (u2 node)][m (u1 node)]
            for (int t = threadIdx.x; t < NQ * GH * np1 * np1; t += blockDim.x) {
                const int v = t / (GH * np1 * np1), r = t % (GH * np1 * np1);
                const int g = r / (np1 * np1), a2 = (r / np1) % np1, mm = r % np1;
                const double* w = gsl >= 0 ? d.gwl + ((int64_t)gsl * GH * d.nc + g * nc) * MAXNP + mm : &T.P2F[0][mm];
                double acc = 0.0;
                for (int ta = 0; ta < nc; ++ta) acc = fma(w[ta * MAXNP], t2b[((v * GH + g) * np1 + a2) * nc + ta], acc);
                t1b[((v * GH + g) * np1 + a2) * np1 + mm] = acc;
            }
            __syncthreads();
            // t1-bar -> node adjoints of (U, J~), then J~(U) at the node
            for (int node = threadIdx.x; node < nn; node += blockDim.x) {
                const int cc[3] = {node % np1, (node / np1) % np1, node / (np1 * np1)};
                const int mm = cc[d2], a1 = cc[u1], a2 = cc[u2];
                double w[NQ];
                for (int v = 0; v < NQ; ++v) {
                    double acc = 0.0;
                    for (int g = 0; g < GH; ++g) {
                        const int cn = s2 ? nc - 1 - g : g;
                        acc = fma(T.P2F[cn][mm], t1b[((v * GH + g) * np1 + a2) * np1 + a1], acc);
                    }
                    w[v] = acc;
                }
                const int64_t pn = (int64_t)nb * d.nn + node;
                double u[NV], ub[NV];
                for (int v = 0; v < NV; ++v) { u[v] = U.dg(v)[pn]; ub[v] = w[v]; }
                current_vjp(u, d.eta, w + NV, w + NV, ub);
                for (int v = 0; v < NV; ++v)
                    if (ub[v] != 0.0) atomicAdd(out.dg(v) + pn, ub[v]);
            }
            __syncthreads();
        } else {
            const int kind = d.bc[e * 6 + f];
            if (kind != FFE_BC_STAR && kind != FFE_BC_NO_INCOMING) continue;
            for (int t = threadIdx.x; t < nper; t += blockDim.x) {
                const int g = t / (nc * nc), ta = t % nc, tb = (t / nc) % nc;
                int c[3];
                c[dd] = s ? nc - 1 : 0;
                c[t1] = ta;
                c[t2] = tb;
                const int64_t p = fdb(d, e) + c[0] + nc * (c[1] + nc * c[2]);
                double ui[NV], u[NV], ub[NV], ib[NV];
                for (int v = 0; v < NV; ++v) { ui[v] = U.fd(v)[p]; ib[v] = 0.0; }
                const ShellPts sp = shell_pts(d, e, nc);
                if (kind == FFE_BC_NO_INCOMING) {
                    double nrm[3];
                    shell_face_normal(sp, dd, s ? nc : 0, ta, tb, nrm);
                    if (!s)
                        for (int qd = 0; qd < 3; ++qd) nrm[qd] = -nrm[qd];
                    bc_no_incoming_flat(ui, nrm, u);
                    ghost_bar(ghost_offset(g, ta, tb), u, ub);
                    bc_no_incoming_vjp(ui, nrm, ub, ib);
                } else {
                    double x[3], ij[3][3];
                    shell_cell(sp, c, ij, x);
                    const double om = omega_of(d, e);
                    bc_star_flat(ui, x, om, u);
                    ghost_bar(ghost_offset(g, ta, tb), u, ub);
                    om_acc += bc_star_vjp(ui, x, om, ub, ib);
                }
                for (int v = 0; v < NV; ++v)
                    if (ib[v] != 0.0) atomicAdd(out.fd(v) + p, ib[v]);
            }
        }
    }
    // Omega-bar: block sum, one atomic per block
    s_om[threadIdx.x] = om_acc;
    __syncthreads();
    if (threadIdx.x == 0 && omega_bar) {
        double acc = 0.0;
        for (int i = 0; i < (int)blockDim.x; ++i) acc += s_om[i];
        if (acc != 0.0) atomicAdd(omega_bar, acc);
    }
}

// Reverse of face_trace: the adjoints the DG reverse mode left at the trace
// nodes of FD faces with a DG neighbour (Dev::ftr_b, [slot][6][12][np1^2]) go
// back through the transposed sum-factorised FD->DG projection -- the two
// tangential directions, then the normal one -- to the 6 cell layers next to
// the face, and through J~(U) at each of those cells, into out.  One CTA per
// (element, face); cells shared by two faces of one element or reached by the
// other FD terms meet in out through FP64 atomics.
__global__ void k_fd_traces_vjp(Dev d, Field U, Field out) {
    extern __shared__ double sm[];
    const int n = d.counts[1];
    const int nfm = d.np1 * d.np1;
    for (int item = blockIdx.x; item < n * 6; item += gridDim.x) {
        const int w = item / 6, f = item % 6;
        const int e = d.fd_list[w];
        const int nb = d.nbr[e * 6 + f];
        if (nb < 0 || d.mask[nb] != 0) continue;
        const ES es = esz(d, e);
        const int np1 = es.np1, nc = es.nc, nc2 = nc * nc;
        const Tables& T = d.tabs[es.P];
        const int dd = f >> 1;
        int t1, t2;
        axes_of(dd, t1, t2);
        const int cn = (f & 1) ? es.P : 0;
        const int lo = T.f2d_lo[cn];
        double* Ob = sm;                          // [12][np1 (t2)][np1 (t1)]
        double* Bb = Ob + NQ * np1 * np1;         // [12][nc (t2)][np1 (t1)]
        double* Ab = Bb + NQ * nc * np1;          // [12][nc (t2)][nc (t1)]
        const double* src = d.ftr_b + ((int64_t)fd_slot_of(d, e) * 6 + f) * NQ * nfm;
        for (int t = threadIdx.x; t < NQ * np1 * np1; t += blockDim.x) {
            const int q = t / (np1 * np1), r = t % (np1 * np1);
            Ob[t] = src[q * nfm + r];
        }
        __syncthreads();
        // t2 direction: Bb[q][b][i] = sum_j F2D[j][b] Ob[q][j][i] (F2D is zero off the stencils)
        for (int t = threadIdx.x; t < NQ * nc * np1; t += blockDim.x) {
            const int q = t / (nc * np1), r = t % (nc * np1);
            const int b = r / np1, i = r % np1;
            double acc = 0.0;
            for (int j = 0; j < np1; ++j) acc = fma(T.F2D[j][b], Ob[(q * np1 + j) * np1 + i], acc);
            Bb[t] = acc;
        }
        __syncthreads();
        // t1 direction: Ab[q][b][a] = sum_i F2D[i][a] Bb[q][b][i]
        for (int t = threadIdx.x; t < NQ * nc2; t += blockDim.x) {
            const int q = t / nc2, r = t % nc2;
            const int b = r / nc, a = r % nc;
            double acc = 0.0;
            for (int i = 0; i < np1; ++i) acc = fma(T.F2D[i][a], Bb[(q * nc + b) * np1 + i], acc);
            Ab[t] = acc;
        }
        __syncthreads();
        // normal direction and the current's chain rule, per cell of the 6 layers
        const int64_t base = fdb(d, e);
        for (int t = threadIdx.x; t < 6 * nc2; t += blockDim.x) {
            const int m = t / nc2, r = t % nc2;
            const double wn = T.F2D[cn][lo + m];
            int c[3];
            c[dd] = lo + m;
            c[t1] = r % nc;
            c[t2] = r / nc;
            const int64_t p = base + c[0] + nc * (c[1] + nc * c[2]);
            double u[NV], ub[NV], jb[3];
            for (int v = 0; v < NV; ++v) {
                u[v] = U.fd(v)[p];
                ub[v] = wn * Ab[v * nc2 + r];
            }
            for (int k = 0; k < 3; ++k) jb[k] = wn * Ab[(NV + k) * nc2 + r];
            current_vjp(u, d.eta, jb, jb, ub);
            for (int v = 0; v < NV; ++v)
                if (ub[v] != 0.0) atomicAdd(out.fd(v) + p, ub[v]);
        }
        __syncthreads();
    }
}

void launch_fd_traces_vjp(const Dev& d, Field U, Field out, cudaStream_t st) {
    if (!d.ftr_b) return;
    const size_t smem = (size_t)(NQ * d.np1 * d.np1 + NQ * d.nc * d.np1 + NQ * d.nc * d.nc) * sizeof(double);
    cudaFuncSetAttribute(k_fd_traces_vjp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    prof_begin("fd_traces_vjp", st);
    k_fd_traces_vjp<<<d.nsm * 2, 256, smem, st>>>(d, U, out);
    prof_end(st);
    g_launch_counter += 1;
}

// out (FD block) must be zeroed and the DG right-hand-side adjoint already
// written by the caller; J holds J~(U) at the FD cells (launch_current).
void launch_fd_rhs_vjp(const Dev& dc, Field U, Field J, Field L, Field out, double* extb, double* gb,
                       double* omega_bar, cudaStream_t st) {
    // chunks of at most FDV_CHUNK elements (fdv_scratch)
    Dev d = dc;
    d.chunk = d.chunk < FDV_CHUNK ? d.chunk : FDV_CHUNK;
    const size_t smem = fdv_ghost_smem(d);
    cudaFuncSetAttribute(k_fdv_ghosts, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    for (int k = 0, nch = fd_chunks(d); k < nch; ++k) {
        const int w0 = k * d.chunk;
        prof_begin("fdv_fill", st);
        launch_fd_fill(d, d.fd_list, 1, w0, U, J, st);
        prof_end(st);
        prof_begin("fdv_lines", st);
        k_fdv_cell_weights<<<d.nsm * 8, 256, 0, st>>>(d, d.fd_list, 1, w0, L, gb);
        k_fdv_lines<<<d.nsm * 8, 64, 0, st>>>(d, d.fd_list, 1, w0, L, gb);
        prof_end(st);
        prof_begin("fdv_gather", st);
        k_fdv_gather<<<d.nsm * 8, 256, 0, st>>>(d, d.fd_list, 1, w0, gb, extb);
        prof_end(st);
        prof_begin("fdv_cells", st);
        k_fdv_cells<<<d.nsm * 8, 256, 0, st>>>(d, d.fd_list, 1, w0, U, L, out, extb);
        prof_end(st);
        prof_begin("fdv_ghosts", st);
        k_fdv_ghosts<<<d.nsm * 2, 256, smem, st>>>(d, d.fd_list, 1, w0, U, J, out, extb, omega_bar);
        prof_end(st);
        g_launch_counter += 5;
    }
}

}  // namespace ffe
