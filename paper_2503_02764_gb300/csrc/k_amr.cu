// Kernels of the composite-grid diffusion solve (fld_amr_*): a coarse block of cells H_d
// with one box refined by 2 in every axis (cells h_d = H_d / 2). The unknowns are the
// coarse cells outside the box and every fine cell; for each, in volume-normalised flux
// form,
//   (A x)_p = x_p + sum_faces c_f (x_p - x_q) + sum_Dirichlet c_w x_p,
//   c_f = dt a_f / V_p,  a_f = (D_p + D_q)/2 * area_f / dist_f,
// with dist_f = H_d (coarse-coarse), h_d (fine-fine), 3 h_d / 2 (a fine cell and the coarse
// cell across the box's edge, one coarse face meeting 2^(d-1) fine faces), and a Dirichlet
// wall at half a cell. Each face flux enters both its cells with opposite signs
// (conservative). Along each axis the box lies strictly inside the block or spans it (then
// the axis's walls apply to the fine cells).
//
// The solve (fld_amr_api.cu) is a two-level scheme: red-black Gauss-Seidel on the
// composite grid (coarse cells, then fine cells, each in two colours), the composite
// residual, its restriction to the whole coarse block (a covered coarse cell takes the
// mean of its fine cells' residuals, the volume-weighted restriction of the flux form),
// the coarse correction by the uniform multigrid solver on the coarse block (covered
// cells carry the mean of their fine cells' D) and its piecewise-constant prolongation.
// FP64 throughout; one thread per cell.
//
// The rows do not change during a solve, and FP64 instructions (above all the divisions of
// every face's conductance) are what the kernels are bound by, so the conductances c_f of the
// faces and the inverse diagonals are formed once per solve (k_amr_weights, k_amr_inverse):
// per grid and axis one array with the extent of that axis one longer than the cells, entry
// i the face below cell i, the last one above the last cell. A face on a wall holds its
// Dirichlet conductance (0 for Neumann) against the value 0; a face between a fine cell and
// the coarse cell outside belongs to the fine grid, and 2^-nd of its conductance couples the
// coarse cell. A colour of a 0.55 M cell grid took 181 us with the rows evaluated in place
// (88 % FP64 pipe).
#include "fld_amr.cuh"
#include "fld_device.cuh"

namespace fld {

namespace {

__device__ __forceinline__ int amr_ncoarse_cells(const AmrGeom& G) {
    return G.nc[0] * G.nc[1] * G.nc[2];
}
__device__ __forceinline__ int amr_nfine_cells(const AmrGeom& G) {
    return G.nf[0] * G.nf[1] * G.nf[2];
}
__device__ __forceinline__ int cidx(const AmrGeom& G, const int* c) {
    return (c[2] * G.nc[1] + c[1]) * G.nc[0] + c[0];
}
__device__ __forceinline__ int fidx(const AmrGeom& G, const int* f) {
    return (f[2] * G.nf[1] + f[1]) * G.nf[0] + f[0];
}
__device__ __forceinline__ bool covered(const AmrGeom& G, const int* c) {
    for (int d = 0; d < G.nd; ++d)
        if (c[d] < G.lo[d] || c[d] >= G.hi[d]) return false;
    return true;
}
__device__ __forceinline__ bool spans(const AmrGeom& G, int d) {
    return G.lo[d] == 0 && G.hi[d] == G.nc[d];
}

// Face value of a Dirichlet wall of the coarse block for coarse cell c (axis d, side s):
// the face array over the two other axes, the lower one fastest.
__device__ __forceinline__ double wall_value(const AmrGeom& G, const double* Ebc, int d, int s,
                                             const int* c) {
    const long long off = G.bcoff[2 * d + s];
    const long long f = d == 0 ? (long long)c[2] * G.nc[1] + c[1]
                      : d == 1 ? (long long)c[2] * G.nc[0] + c[0]
                               : (long long)c[1] * G.nc[0] + c[0];
    return Ebc[off + f];
}

// Operator row of coarse cell c (uncovered): diag = 1 + sum c_f (+ walls), off = sum c_f x_q,
// wall = sum c_w E_b (the right-hand side's wall term).
__device__ void coarse_row(const AmrGeom& G, const double* Dc, const double* Df,
                           const double* xc, const double* xf, const double* Ebc, const int* c,
                           double& diag, double& off, double& wall) {
    const double Dp = Dc[cidx(G, c)];
    diag = 1.0;
    off = 0.0;
    wall = 0.0;
    for (int d = 0; d < G.nd; ++d) {
        const double H2 = G.H[d] * G.H[d];
        for (int s = 0; s < 2; ++s) {
            int q[3] = {c[0], c[1], c[2]};
            q[d] += s ? 1 : -1;
            if (q[d] < 0 || q[d] >= G.nc[d]) {
                const int kind = s ? G.bchi[d] : G.bclo[d];
                if (kind == FLD_BC_PERIODIC) {
                    q[d] = (q[d] + G.nc[d]) % G.nc[d];
                } else {
                    if (kind == FLD_BC_DIRICHLET) {
                        const double cw = G.dt * 2.0 * Dp / H2;
                        diag += cw;
                        if (Ebc) wall += cw * wall_value(G, Ebc, d, s, c);
                    }
                    continue;
                }
            }
            if (!covered(G, q)) {
                const double cf = G.dt * 0.5 * (Dp + Dc[cidx(G, q)]) / H2;
                diag += cf;
                off += cf * xc[cidx(G, q)];
                continue;
            }
            // the box's edge: the 2^(nd-1) fine cells of the layer facing c
            int f0[3] = {0, 0, 0};
            for (int e = 0; e < G.nd; ++e) f0[e] = 2 * (c[e] - G.lo[e]);
            f0[d] = s ? 0 : G.nf[d] - 1;
            const double w = G.dt * 0.5 / (0.75 * H2 * (double)(1 << (G.nd - 1)));
            const int t1 = d == 0 ? 1 : 0, t2 = d == 2 ? 1 : 2;
            const int n1 = t1 < G.nd ? 2 : 1, n2 = t2 < G.nd ? 2 : 1;
            for (int b = 0; b < n2; ++b)
                for (int a = 0; a < n1; ++a) {
                    int f[3] = {f0[0], f0[1], f0[2]};
                    f[t1] += a;
                    f[t2] += b;
                    const int fi = fidx(G, f);
                    const double cf = w * (Dp + Df[fi]);
                    diag += cf;
                    off += cf * xf[fi];
                }
        }
    }
}

// Operator row of fine cell f.
__device__ void fine_row(const AmrGeom& G, const double* Dc, const double* Df, const double* xc,
                         const double* xf, const double* Ebc, const int* f, double& diag,
                         double& off, double& wall) {
    const double Dp = Df[fidx(G, f)];
    diag = 1.0;
    off = 0.0;
    wall = 0.0;
    for (int d = 0; d < G.nd; ++d) {
        const double h2 = 0.25 * G.H[d] * G.H[d];
        for (int s = 0; s < 2; ++s) {
            int g[3] = {f[0], f[1], f[2]};
            g[d] += s ? 1 : -1;
            if (g[d] >= 0 && g[d] < G.nf[d]) {
                const double cf = G.dt * 0.5 * (Dp + Df[fidx(G, g)]) / h2;
                diag += cf;
                off += cf * xf[fidx(G, g)];
                continue;
            }
            if (spans(G, d)) {
                const int kind = s ? G.bchi[d] : G.bclo[d];
                if (kind == FLD_BC_PERIODIC) {
                    g[d] = (g[d] + G.nf[d]) % G.nf[d];
                    const double cf = G.dt * 0.5 * (Dp + Df[fidx(G, g)]) / h2;
                    diag += cf;
                    off += cf * xf[fidx(G, g)];
                } else if (kind == FLD_BC_DIRICHLET) {
                    const double cw = G.dt * 2.0 * Dp / h2;
                    diag += cw;
                    if (Ebc) {
                        int c[3] = {0, 0, 0};
                        for (int e = 0; e < 3; ++e) c[e] = e < G.nd ? G.lo[e] + f[e] / 2 : 0;
                        wall += cw * wall_value(G, Ebc, d, s, c);
                    }
                }
                continue;
            }
            // the coarse cell across the box's edge
            int c[3] = {0, 0, 0};
            for (int e = 0; e < 3; ++e) c[e] = e < G.nd ? G.lo[e] + f[e] / 2 : 0;
            c[d] += s ? 1 : -1;
            const int ci = cidx(G, c);
            const double cf = G.dt * 0.5 * (Dp + Dc[ci]) / (1.5 * h2);
            diag += cf;
            off += cf * xc[ci];
        }
    }
}

__device__ __forceinline__ void coarse_coord(const AmrGeom& G, int p, int* c) {
    c[0] = p % G.nc[0];
    const int q = p / G.nc[0];
    c[1] = q % G.nc[1];
    c[2] = q / G.nc[1];
}
__device__ __forceinline__ void fine_coord(const AmrGeom& G, int p, int* f) {
    f[0] = p % G.nf[0];
    const int q = p / G.nf[0];
    f[1] = q % G.nf[1];
    f[2] = q / G.nf[1];
}

// b = E + wall terms (unknown cells); DH = Dc (uncovered) or the mean of the fine D
__global__ void k_amr_setup(AmrGeom G, const double* __restrict__ Dc,
                            const double* __restrict__ Df, const double* __restrict__ Ec,
                            const double* __restrict__ Ef, const double* __restrict__ Ebc,
                            double* __restrict__ bc, double* __restrict__ bf,
                            double* __restrict__ DH) {
    const int nC = amr_ncoarse_cells(G), nF = amr_nfine_cells(G);
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < nC + nF; p += gridDim.x * blockDim.x) {
        double diag, off, wall;
        if (p < nC) {
            int c[3];
            coarse_coord(G, p, c);
            if (covered(G, c)) {
                double s = 0.0;
                const int n1 = G.nd > 1 ? 2 : 1, n2 = G.nd > 2 ? 2 : 1;
                for (int z = 0; z < n2; ++z)
                    for (int y = 0; y < n1; ++y)
                        for (int x = 0; x < 2; ++x) {
                            const int f[3] = {2 * (c[0] - G.lo[0]) + x,
                                              G.nd > 1 ? 2 * (c[1] - G.lo[1]) + y : 0,
                                              G.nd > 2 ? 2 * (c[2] - G.lo[2]) + z : 0};
                            s += Df[fidx(G, f)];
                        }
                DH[p] = s / (double)(2 * n1 * n2);
                bc[p] = 0.0;
            } else {
                coarse_row(G, Dc, Df, Ec, Ef, Ebc, c, diag, off, wall);
                DH[p] = Dc[p];
                bc[p] = Ec[p] + wall;
            }
        } else {
            int f[3];
            fine_coord(G, p - nC, f);
            fine_row(G, Dc, Df, Ec, Ef, Ebc, f, diag, off, wall);
            bf[p - nC] = Ef[p - nC] + wall;
        }
    }
}

// ---- stored rows: face conductances and inverse diagonals of one grid
template <bool FINE>
__device__ __forceinline__ const int* extents(const AmrGeom& G) { return FINE ? G.nf : G.nc; }

// index of the face below cell (c0, c1, c2) along axis d; the one above is `step` further
// (unsigned: below 2^31 cells have up to twice as many faces along an axis)
__device__ __forceinline__ unsigned face_at(const int* n, int d, const int* c, unsigned& step) {
    const unsigned nx = n[0], ny = n[1], x = c[0], y = c[1], z = c[2];
    step = d == 0 ? 1u : d == 1 ? nx : nx * ny;
    return d == 0   ? (z * ny + y) * (nx + 1u) + x
           : d == 1 ? (z * (ny + 1u) + y) * nx + x
                    : (z * ny + y) * nx + x;
}

// conductance of the face below (s = 0) or above (s = 1) the cell, as its grid stores it
template <bool FINE>
__device__ double conductance(const AmrGeom& G, const double* Dc, const double* Df, const int* c,
                              int d, int s) {
    const int* n = extents<FINE>(G);
    const double* D = FINE ? Df : Dc;
    const double h2 = (FINE ? 0.25 : 1.0) * G.H[d] * G.H[d];
    if (!FINE && covered(G, c)) return 0.0;
    const double Dp = D[FINE ? fidx(G, c) : cidx(G, c)];
    int q[3] = {c[0], c[1], c[2]};
    q[d] += s ? 1 : -1;
    if (q[d] < 0 || q[d] >= n[d]) {
        if (FINE && !spans(G, d)) {
            int o[3] = {0, 0, 0};
            for (int e = 0; e < G.nd; ++e) o[e] = G.lo[e] + c[e] / 2;
            o[d] += s ? 1 : -1;
            return G.dt * 0.5 * (Dp + Dc[cidx(G, o)]) / (1.5 * h2);
        }
        const int kind = s ? G.bchi[d] : G.bclo[d];
        if (kind != FLD_BC_PERIODIC) return kind == FLD_BC_DIRICHLET ? G.dt * 2.0 * Dp / h2 : 0.0;
        q[d] = (q[d] + n[d]) % n[d];
    }
    if (!FINE && covered(G, q)) return 0.0;
    return G.dt * 0.5 * (Dp + D[FINE ? fidx(G, q) : cidx(G, q)]) / h2;
}

template <bool FINE>
__global__ void k_amr_weights(AmrGeom G, AmrRows R, const double* __restrict__ Dc,
                              const double* __restrict__ Df) {
    const int* n = extents<FINE>(G);
    const int cells = FINE ? amr_nfine_cells(G) : amr_ncoarse_cells(G);
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < cells; p += gridDim.x * blockDim.x) {
        int c[3];
        if (FINE) fine_coord(G, p, c);
        else coarse_coord(G, p, c);
        for (int d = 0; d < G.nd; ++d) {
            unsigned step;
            const unsigned f = face_at(n, d, c, step);
            R.w[d][f] = conductance<FINE>(G, Dc, Df, c, d, 0);
            if (c[d] == n[d] - 1) R.w[d][f + step] = conductance<FINE>(G, Dc, Df, c, d, 1);
        }
    }
}

// A cell of one grid with its faces. visit(w, x) sees every face's conductance and the value
// across it (0 beyond a wall).
template <bool FINE, typename F>
__device__ __forceinline__ void faces(const AmrGeom& G, const AmrRows& Rc, const AmrRows& Rf,
                                      const double* xc, const double* xf, const int* c, int p,
                                      F&& visit) {
    const int* n = extents<FINE>(G);
    const double* x = FINE ? xf : xc;
    const int stride[3] = {1, n[0], n[0] * n[1]};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        if (d >= G.nd) break;
        unsigned step;
        const unsigned f = face_at(n, d, c, step);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const double w = (FINE ? Rf : Rc).w[d][f + (s ? step : 0u)];
            const bool edge = s ? c[d] == n[d] - 1 : c[d] == 0;
            int q = s ? p + stride[d] : p - stride[d];
            if (edge) {
                if (FINE && !spans(G, d)) {            // the coarse cell outside the box
                    int o[3] = {0, 0, 0};
                    for (int e = 0; e < 3; ++e) o[e] = e < G.nd ? G.lo[e] + c[e] / 2 : 0;
                    o[d] += s ? 1 : -1;
                    visit(w, xc[cidx(G, o)]);
                    continue;
                }
                if ((s ? G.bchi[d] : G.bclo[d]) != FLD_BC_PERIODIC) {
                    visit(w, 0.0);
                    continue;
                }
                q = s ? p - (n[d] - 1) * stride[d] : p + (n[d] - 1) * stride[d];
            }
            if (!FINE) {
                int o[3] = {c[0], c[1], c[2]};
                o[d] = s ? (edge ? 0 : c[d] + 1) : (edge ? n[d] - 1 : c[d] - 1);
                if (covered(G, o)) {                   // the box: the fine cells facing c
                    int f0[3] = {0, 0, 0};
                    for (int e = 0; e < G.nd; ++e) f0[e] = 2 * (c[e] - G.lo[e]);
                    f0[d] = s ? 0 : G.nf[d] - 1;
                    const double part = G.nd == 3 ? 0.125 : G.nd == 2 ? 0.25 : 0.5;
                    const int t1 = d == 0 ? 1 : 0, t2 = d == 2 ? 1 : 2;
                    const int n1 = t1 < G.nd ? 2 : 1, n2 = t2 < G.nd ? 2 : 1;
                    for (int b = 0; b < n2; ++b)
                        for (int a = 0; a < n1; ++a) {
                            int g[3] = {f0[0], f0[1], f0[2]};
                            g[t1] += a;
                            g[t2] += b;
                            unsigned st;
                            const unsigned fg = face_at(G.nf, d, g, st);
                            visit(part * Rf.w[d][s ? fg : fg + st], xf[fidx(G, g)]);
                        }
                    continue;
                }
            }
            visit(w, x[q]);
        }
    }
}

template <bool FINE>
__global__ void k_amr_inverse(AmrGeom G, AmrRows Rc, AmrRows Rf, const double* __restrict__ xc,
                              const double* __restrict__ xf) {
    const int cells = FINE ? amr_nfine_cells(G) : amr_ncoarse_cells(G);
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < cells; p += gridDim.x * blockDim.x) {
        int c[3];
        if (FINE) fine_coord(G, p, c);
        else coarse_coord(G, p, c);
        double dg = 1.0;
        if (FINE || !covered(G, c))
            faces<FINE>(G, Rc, Rf, xc, xf, c, p, [&](double w, double) { dg += w; });
        (FINE ? Rf : Rc).inv[p] = 1.0 / dg;
    }
}

// One colour of one grid, one thread per pair of cells along x.
template <bool FINE>
__global__ void __launch_bounds__(256)
k_amr_smooth(AmrGeom G, AmrRows Rc, AmrRows Rf, int colour, const double* __restrict__ b,
             double* xc, double* xf) {
    after_previous();
    const int* n = extents<FINE>(G);
    for (int k = blockIdx.z; k < n[2]; k += gridDim.z)
        for (int j = blockIdx.y * blockDim.y + threadIdx.y; j < n[1]; j += gridDim.y * blockDim.y) {
            const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x) + ((j + k + colour) & 1);
            if (i >= n[0]) continue;
            const int c[3] = {i, j, k};
            if (!FINE && covered(G, c)) continue;
            const int p = (k * n[1] + j) * n[0] + i;
            double s = b[p];
            faces<FINE>(G, Rc, Rf, xc, xf, c, p, [&](double w, double v) { s = fma(w, v, s); });
            (FINE ? xf : xc)[p] = s * (FINE ? Rf : Rc).inv[p];
        }
}

// r = b - A x over the unknowns of one grid (differences first), and partial sums of r^2
template <bool FINE>
__global__ void __launch_bounds__(256)
k_amr_resid(AmrGeom G, AmrRows Rc, AmrRows Rf, const double* __restrict__ b,
            const double* __restrict__ xc, const double* __restrict__ xf,
            double* __restrict__ r, double* __restrict__ partials, double one) {
    after_previous();
    __shared__ double sh[32];
    const int* n = extents<FINE>(G);
    const int lx = threadIdx.x & 31, ly = threadIdx.x >> 5;
    const int ntx = (n[0] + 31) / 32, nty = (n[1] + 7) / 8;
    const int tiles = ntx * nty * n[2];
    double acc = 0.0;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int q = t / ntx, k = q / nty;
        const int i = (t - q * ntx) * 32 + lx, j = (q - k * nty) * 8 + ly;
        if (i >= n[0] || j >= n[1]) continue;
        const int c[3] = {i, j, k};
        if (!FINE && covered(G, c)) continue;
        const int p = (k * n[1] + j) * n[0] + i;
        const double x = (FINE ? xf : xc)[p];
        double v = fma(x, -one, b[p]);
        faces<FINE>(G, Rc, Rf, xc, xf, c, p,
                    [&](double w, double xq) { v = fma(w, fma(x, -one, xq), v); });
        r[p] = v;
        acc = fma(v, v, acc);
    }
    acc = block_sum(acc, sh);
    if (threadIdx.x == 0) partials[blockIdx.x] = acc;
}

// covered coarse cells: the mean of their fine cells (of v)
__global__ void k_amr_average(AmrGeom G, const double* __restrict__ vf, double* vc) {
    after_previous();
    const int nC = amr_ncoarse_cells(G);
    const int n1 = G.nd > 1 ? 2 : 1, n2 = G.nd > 2 ? 2 : 1;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < nC; p += gridDim.x * blockDim.x) {
        int c[3];
        coarse_coord(G, p, c);
        if (!covered(G, c)) continue;
        double s = 0.0;
        for (int z = 0; z < n2; ++z)
            for (int y = 0; y < n1; ++y)
                for (int x = 0; x < 2; ++x) {
                    const int f[3] = {2 * (c[0] - G.lo[0]) + x,
                                      G.nd > 1 ? 2 * (c[1] - G.lo[1]) + y : 0,
                                      G.nd > 2 ? 2 * (c[2] - G.lo[2]) + z : 0};
                    s += vf[fidx(G, f)];
                }
        vc[p] = s / (double)(2 * n1 * n2);
    }
}

// x += e on the composite grid: uncovered coarse cells directly, fine cells from their
// parent (piecewise constant)
__global__ void k_amr_correct(AmrGeom G, const double* __restrict__ e, double* xc, double* xf) {
    after_previous();
    const int nC = amr_ncoarse_cells(G), nF = amr_nfine_cells(G);
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < nC + nF; p += gridDim.x * blockDim.x) {
        if (p < nC) {
            int c[3];
            coarse_coord(G, p, c);
            if (!covered(G, c)) xc[p] += e[p];
        } else {
            int f[3];
            fine_coord(G, p - nC, f);
            int c[3] = {0, 0, 0};
            for (int d = 0; d < 3; ++d) c[d] = d < G.nd ? G.lo[d] + f[d] / 2 : 0;
            xf[p - nC] += e[cidx(G, c)];
        }
    }
}

int amr_blocks(long long n) {
    const long long nb = (n + 255) / 256;
    return (int)std::max<long long>(1, std::min<long long>(nb, (long long)num_sms() * 16));
}

}  // namespace

void launch_amr_setup(const AmrGeom& G, const double* Dc, const double* Df, const double* Ec,
                      const double* Ef, const double* Ebc, double* bc, double* bf, double* DH,
                      cudaStream_t s) {
    const long long n = (long long)G.nc[0] * G.nc[1] * G.nc[2] + (long long)G.nf[0] * G.nf[1] * G.nf[2];
    k_amr_setup<<<amr_blocks(n), 256, 0, s>>>(G, Dc, Df, Ec, Ef, Ebc, bc, bf, DH);
}

void launch_amr_rows(const AmrGeom& G, const AmrRows& Rc, const AmrRows& Rf, const double* Dc,
                     const double* Df, const double* xc, const double* xf, cudaStream_t s) {
    const int bc = amr_blocks((long long)G.nc[0] * G.nc[1] * G.nc[2]);
    const int bf = amr_blocks((long long)G.nf[0] * G.nf[1] * G.nf[2]);
    k_amr_weights<false><<<bc, 256, 0, s>>>(G, Rc, Dc, Df);
    k_amr_weights<true><<<bf, 256, 0, s>>>(G, Rf, Dc, Df);
    k_amr_inverse<false><<<bc, 256, 0, s>>>(G, Rc, Rf, xc, xf);
    k_amr_inverse<true><<<bf, 256, 0, s>>>(G, Rc, Rf, xc, xf);
}

void launch_amr_smooth(const AmrGeom& G, const AmrRows& Rc, const AmrRows& Rf, int phase,
                       const double* bc, const double* bf, double* xc, double* xf,
                       cudaStream_t s) {
    const int* n = phase >= 2 ? G.nf : G.nc;
    const int pairs = (n[0] + 1) / 2;
    const dim3 blk = pairs > 16 ? dim3(32, 8) : dim3(16, 16);
    const dim3 grd((pairs + blk.x - 1) / blk.x, std::min<int>((n[1] + blk.y - 1) / blk.y, 65535),
                   std::min(n[2], 65535));
    if (phase >= 2) launch_chained(true, k_amr_smooth<true>, grd, blk, 0, s, G, Rc, Rf, phase & 1,
                                   bf, xc, xf);
    else launch_chained(true, k_amr_smooth<false>, grd, blk, 0, s, G, Rc, Rf, phase & 1, bc, xc,
                        xf);
}

// two launches; returns the partial sums written (<= nblocks)
int launch_amr_resid(const AmrGeom& G, const AmrRows& Rc, const AmrRows& Rf, const double* bc,
                     const double* bf, const double* xc, const double* xf, double* rc, double* rf,
                     double* partials, int nblocks, cudaStream_t s) {
    auto blocks = [&](const int* n) {
        const long long t = (long long)((n[0] + 31) / 32) * ((n[1] + 7) / 8) * n[2];
        return (int)std::min<long long>(t, nblocks / 2);
    };
    const int nc = blocks(G.nc), nf = blocks(G.nf);
    launch_chained(true, k_amr_resid<false>, nc, 256, 0, s, G, Rc, Rf, bc, xc, xf, rc, partials,
                   1.0);
    launch_chained(true, k_amr_resid<true>, nf, 256, 0, s, G, Rc, Rf, bf, xc, xf, rf, partials + nc,
                   1.0);
    return nc + nf;
}

void launch_amr_average(const AmrGeom& G, const double* vf, double* vc, cudaStream_t s) {
    launch_chained(true, k_amr_average, amr_blocks((long long)G.nc[0] * G.nc[1] * G.nc[2]), 256, 0,
                   s, G, vf, vc);
}

void launch_amr_correct(const AmrGeom& G, const double* e, double* xc, double* xf,
                        cudaStream_t s) {
    const long long n = (long long)G.nc[0] * G.nc[1] * G.nc[2] + (long long)G.nf[0] * G.nf[1] * G.nf[2];
    launch_chained(true, k_amr_correct, amr_blocks(n), 256, 0, s, G, e, xc, xf);
}

}  // namespace fld
