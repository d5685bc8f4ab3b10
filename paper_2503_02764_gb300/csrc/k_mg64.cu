// FP64 V-cycle kernels of 2D and 3D levels on stored coefficients.
//
// FP64 instructions bound these kernels, not memory: this GPU issues 0.5 T of them a second
// (19.2 cycles of an SM a warp), some 75 times fewer than FP32 ones. Evaluating the face
// coefficients from K in every half sweep took about 40 FP64 instructions per updated cell (six
// sums, six weightings, the diagonal and a division): 651 us per half sweep of a 256^3 level. The
// coefficients do not change during a solve, so they are formed once per level and solve:
//   wx, wy, wz  the weight mean(K_p, K_q) w_d of the face towards the lower neighbour along
//               each axis (the wrapped face for the first cell of a periodic axis; 0 at walls),
//   inv         1 / (1 + the six weights + 2 K w_d per Dirichlet face),
// and a relaxation is x_p = (b_p + sum w x_q) inv_p: seven FP64 instructions. The kernel then
// moves 56 B a cell (b, inv, x twice, three weights; the two colours share every sector) in
// place of 32, which is the cheaper side.
//
// The arrays live in the buffers of the mixed modes (the double-FP32 pairs on the finest
// level, the FP32 pyramid below it), which an FP64 solve does not use.
#include <algorithm>

#include "fld_device.cuh"

namespace fld {

namespace {

struct Nb {          // neighbour indices along an axis, -1 beyond a wall
    int lo, hi;
};

__device__ __forceinline__ Nb axis_nb(int c, int n, int p, int stride, bool per) {
    Nb r;
    r.lo = c > 0 ? p - stride : (per ? p + (n - 1) * stride : -1);
    r.hi = c < n - 1 ? p + stride : (per ? p - (n - 1) * stride : -1);
    return r;
}

// the neighbours of cell (i, j, k); the face towards nb.hi has its weight stored there
template <int ND>
__device__ __forceinline__ void cell_nb(const Lvl& L, int i, int j, int k, int p, Nb nb[3]) {
    const int nx = L.n[0], ny = L.n[1];
    nb[0] = axis_nb(i, nx, p, 1, L.bclo[0] == FLD_BC_PERIODIC);
    nb[1] = axis_nb(j, ny, p, nx, L.bclo[1] == FLD_BC_PERIODIC);
    if (ND == 3) nb[2] = axis_nb(k, L.n[2], p, nx * ny, L.bclo[2] == FLD_BC_PERIODIC);
}

template <int ND>
__global__ void __launch_bounds__(256)
k_coef64(Lvl L, double3 half, const double* __restrict__ K, Coef64 W, double one) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= L.n[0] || j >= L.n[1]) return;
    const int p = (int)fld_at(((long long)k * L.n[1] + j) * L.n[0] + i, L.ncell);
    const double kc = K[p];
    Nb nb[3];
    cell_nb<ND>(L, i, j, k, p, nb);
    double sw = 1.0;
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        const double hd = d == 0 ? half.x : d == 1 ? half.y : half.z, dw = L.w[d];
        // the sum of two cells' K
        auto ksum = [&](int q) { return L.fm ? fsum2(kc, K[q], 1) : fma(K[q], one, kc); };
        double w = 0.0;
        if (nb[d].lo >= 0) {
            w = ksum(nb[d].lo) * hd;
            sw = fma(w, one, sw);
        } else if (L.bclo[d] == FLD_BC_DIRICHLET) {
            sw = fma(2.0 * kc, dw, sw);
        }
        (d == 0 ? W.wx : d == 1 ? W.wy : W.wz)[p] = w;
        if (nb[d].hi >= 0) sw = fma(ksum(nb[d].hi), hd, sw);
        else if (L.bchi[d] == FLD_BC_DIRICHLET) sw = fma(2.0 * kc, dw, sw);
    }
    W.inv[p] = in_f32_range(sw) ? rcp_nr(sw) : 1.0 / sw;
}

// b + sum over the faces of w x_q
template <int ND>
__device__ __forceinline__ double gather64(const Nb nb[3], int p, const Coef64& W,
                                           const double* __restrict__ x, double s) {
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        const double* __restrict__ w = d == 0 ? W.wx : d == 1 ? W.wy : W.wz;
        if (nb[d].lo >= 0) s = fma(w[p], x[nb[d].lo], s);
        if (nb[d].hi >= 0) s = fma(w[nb[d].hi], x[nb[d].hi], s);
    }
    return s;
}

// Red-black half sweep: one thread per pair of cells along x, the one of `color` relaxed.
// In place where no periodic extent is odd; otherwise (OOP) from xin to xout, the other
// colour copied, so that two same-colour cells that meet across the wrap do not race.
// 256^3: 651 us with the coefficients evaluated from K, 136 us here (6.9 TB/s of the 56 B a
// cell; 98 us of FP64 issue).
template <int ND, bool OOP>
__global__ void __launch_bounds__(256)
k_half64(Lvl L, int color, const double* xin, double* xout, const double* __restrict__ b,
         Coef64 W) {
    after_previous();
    const int ip = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    if (j >= L.n[1]) return;
    const int par = (j + k + color) & 1;
    const int i = 2 * ip + par;
    const int row = (int)(((long long)k * L.n[1] + j) * L.n[0]);
    if (OOP) {
        const int o = 2 * ip + (par ^ 1);
        if (o < L.n[0]) xout[fld_at(row + o, L.ncell)] = xin[row + o];
    }
    if (i >= L.n[0]) return;
    const int p = (int)fld_at(row + i, L.ncell);
    Nb nb[3];
    cell_nb<ND>(L, i, j, k, p, nb);
    xout[p] = gather64<ND>(nb, p, W, xin, b[p]) * W.inv[p];
}

// r = b - x - sum_faces w (x - x_q) - sum_Dirichlet 2 K w_d x: differences first, so that the
// rounding scales with the fluxes and not with the weights
template <int ND>
__device__ __forceinline__ double resid_cell64(const Lvl& L, const Nb nb[3], int p,
                                               const Coef64& W, const double* __restrict__ x,
                                               const double* __restrict__ b,
                                               const double* __restrict__ K, double one) {
    const double xc = x[p];
    double r = fma(xc, -one, b[p]);
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        const double* __restrict__ w = d == 0 ? W.wx : d == 1 ? W.wy : W.wz;
        if (nb[d].lo >= 0) r = fma(w[p], fma(xc, -one, x[nb[d].lo]), r);
        else if (L.bclo[d] == FLD_BC_DIRICHLET) r = fma(-2.0 * L.w[d] * K[p], xc, r);
        if (nb[d].hi >= 0) r = fma(w[nb[d].hi], fma(xc, -one, x[nb[d].hi]), r);
        else if (L.bchi[d] == FLD_BC_DIRICHLET) r = fma(-2.0 * L.w[d] * K[p], xc, r);
    }
    return r;
}

// Partial sums of the squared residual: fourteen FP64 instructions a cell (256^3: 451 us, 882 us
// with the six face sums evaluated here).
template <int ND>
__global__ void __launch_bounds__(256)
k_norm64(Lvl L, const double* __restrict__ x, const double* __restrict__ b,
         const double* __restrict__ K, Coef64 W, double* __restrict__ partials, int tx, int ty,
         double one) {
    after_previous();
    __shared__ double sh[32];
    double a2 = 0.0;
    const int ntx = (L.n[0] + tx - 1) / tx, nty = (L.n[1] + ty - 1) / ty;
    const int lx = threadIdx.x % tx, ly = threadIdx.x / tx;
    const int tiles = ntx * nty * L.n[2];      // no more than the cells, below 2^31
    for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int q = t / ntx;
        const int i = (t - q * ntx) * tx + lx;
        const int k = q / nty, j = (q - k * nty) * ty + ly;
        if (i >= L.n[0] || j >= L.n[1]) continue;
        const int p = (int)fld_at(((long long)k * L.n[1] + j) * L.n[0] + i, L.ncell);
        Nb nb[3];
        cell_nb<ND>(L, i, j, k, p, nb);
        const double r = resid_cell64<ND>(L, nb, p, W, x, b, K, one);
        a2 = fma(r, r, a2);
    }
    a2 = block_sum(a2, sh);
    if (threadIdx.x == 0) partials[blockIdx.x] = a2;
}

// Coarse right-hand side: the mean of the children's residuals. RED (3D, every axis halved
// exactly, after a red-black sweep): only the four red children, whose siblings' residuals
// vanish up to the rounding of their relaxation.
template <int ND, bool RED>
__global__ void __launch_bounds__(128)
k_restrict64(Lvl F, Lvl C, const double* __restrict__ x, const double* __restrict__ b,
             const double* __restrict__ K, Coef64 W, double* __restrict__ bc, double one) {
    after_previous();
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = blockIdx.y * blockDim.y + threadIdx.y;
    const int Kc = blockIdx.z;
    if (I >= C.n[0] || J >= C.n[1]) return;
    double s = 0.0;
    if (RED) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int dj = c & 1, dk = c >> 1;
            const int i = 2 * I + (dj ^ dk), j = 2 * J + dj, k = 2 * Kc + dk;
            const int p = (int)fld_at(((long long)k * F.n[1] + j) * F.n[0] + i, F.ncell);
            Nb nb[3];
            cell_nb<ND>(F, i, j, k, p, nb);
            s = fma(resid_cell64<ND>(F, nb, p, W, x, b, K, one), one, s);
        }
        s *= 0.125;
    } else {
        const int ci[3] = {I, J, Kc};
        int lo[3], hi[3], cnt = 1;
        for (int d = 0; d < 3; ++d) {
            lo[d] = C.n[d] < F.n[d] ? 2 * ci[d] : ci[d];
            hi[d] = C.n[d] < F.n[d] ? min(2 * ci[d] + 1, F.n[d] - 1) : ci[d];
            cnt *= hi[d] - lo[d] + 1;
        }
        for (int k = lo[2]; k <= hi[2]; ++k)
            for (int j = lo[1]; j <= hi[1]; ++j)
                for (int i = lo[0]; i <= hi[0]; ++i) {
                    const int p = (int)fld_at(((long long)k * F.n[1] + j) * F.n[0] + i, F.ncell);
                    Nb nb[3];
                    cell_nb<ND>(F, i, j, k, p, nb);
                    s = fma(resid_cell64<ND>(F, nb, p, W, x, b, K, one), one, s);
                }
        s *= cnt == 8 ? 0.125 : cnt == 4 ? 0.25 : cnt == 2 ? 0.5 : 1.0;
    }
    bc[fld_at(((long long)Kc * C.n[1] + J) * C.n[0] + I, C.ncell)] = s;
}

dim3 rows_block(int n) { return n > 16 ? dim3(32, 8) : dim3(16, 16); }

dim3 rows_grid64(const Lvl& L, int nx, dim3 blk) {
    return dim3((nx + blk.x - 1) / blk.x, (L.n[1] + blk.y - 1) / blk.y, L.n[2]);
}

}  // namespace

// grids whose y and z extents fit a launch grid; the rest keep the kernels on K
bool mg64_ok(const Lvl& L) {
    return L.ndim >= 2 && L.n[1] <= 65535 && L.n[2] <= 65535;
}

void launch_coef64(const Lvl& L, const double* K, const Coef64& W, cudaStream_t s) {
    const dim3 blk = rows_block(L.n[0]), grd = rows_grid64(L, L.n[0], blk);
    const double3 half = make_double3(0.5 * L.w[0], 0.5 * L.w[1], 0.5 * L.w[2]);
    if (L.ndim == 3) k_coef64<3><<<grd, blk, 0, s>>>(L, half, K, W, 1.0);
    else k_coef64<2><<<grd, blk, 0, s>>>(L, half, K, W, 1.0);
}

void launch_half64(const Lvl& L, int color, const double* xin, double* xout, const double* b,
                   const Coef64& W, cudaStream_t s) {
    const int pairs = (L.n[0] + 1) / 2;
    const dim3 blk = rows_block(pairs), grd = rows_grid64(L, pairs, blk);
    if (xin == xout) {
        if (L.ndim == 3) launch_chained(true, k_half64<3, false>, grd, blk, 0, s, L, color, xin,
                                        xout, b, W);
        else launch_chained(true, k_half64<2, false>, grd, blk, 0, s, L, color, xin, xout, b, W);
    } else {
        if (L.ndim == 3) launch_chained(true, k_half64<3, true>, grd, blk, 0, s, L, color, xin,
                                        xout, b, W);
        else launch_chained(true, k_half64<2, true>, grd, blk, 0, s, L, color, xin, xout, b, W);
    }
}

int launch_norm64(const Lvl& L, const double* x, const double* b, const double* K,
                  const Coef64& W, double* partials, int nblocks, cudaStream_t s) {
    const int tx = L.n[0] > 16 ? 32 : 16, ty = 256 / tx;
    const long long tiles = (long long)((L.n[0] + tx - 1) / tx) * ((L.n[1] + ty - 1) / ty) * L.n[2];
    const int nb = (int)std::min<long long>(tiles, nblocks);
    if (L.ndim == 3) launch_chained(true, k_norm64<3>, nb, 256, 0, s, L, x, b, K, W, partials, tx,
                                    ty, 1.0);
    else launch_chained(true, k_norm64<2>, nb, 256, 0, s, L, x, b, K, W, partials, tx, ty, 1.0);
    return nb;
}

void launch_restrict64(const Lvl& F, const Lvl& C, const double* x, const double* b,
                       const double* K, const Coef64& W, double* bc, bool red_only,
                       cudaStream_t s) {
    const dim3 blk = C.n[0] > 16 ? dim3(32, 4) : dim3(8, 16);
    const dim3 grd((C.n[0] + blk.x - 1) / blk.x, (C.n[1] + blk.y - 1) / blk.y, C.n[2]);
    if (F.ndim == 3) {
        if (red_only && transfer3_ok(F, C))
            launch_chained(true, k_restrict64<3, true>, grd, blk, 0, s, F, C, x, b, K, W, bc, 1.0);
        else
            launch_chained(true, k_restrict64<3, false>, grd, blk, 0, s, F, C, x, b, K, W, bc, 1.0);
    } else {
        launch_chained(true, k_restrict64<2, false>, grd, blk, 0, s, F, C, x, b, K, W, bc, 1.0);
    }
}

}  // namespace fld
