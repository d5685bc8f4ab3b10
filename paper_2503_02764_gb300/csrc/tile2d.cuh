// A tile of a 2D FP32 multigrid level in shared memory: (prolongation +) n red-black sweeps
// (+ residual and restriction), out of place. Shared by the single-grid V-cycle (k_tile2d.cu)
// and the batched step (batch_step.cuh).
//
// The tile is loaded with a halo of H cells, and every half sweep relaxes a region one cell
// smaller on each side (the halo's values are recomputed, not exchanged between tiles): H = 2 n,
// one more where the residual of the tile follows. The updates are those of the half-sweep
// kernels, cell for cell, since a cell of one colour reads only the other colour. On an odd
// periodic extent two cells of one colour meet across the wrap: there a half sweep reads one
// copy of x and writes another, as the out-of-place half sweeps do.
//
// The loaded region is T2_W = 64 columns wide: 32 pairs, so that a warp relaxes the cells of one
// colour in a row with every lane, and a lane's columns (and their interpolation weights) are the
// same in every row. The kernel is bound by instruction issue (~45 a relaxation, most of them
// shared-memory reads and the face sums); with rows of 74 columns, 58 % of the lanes at work and
// the column's index arithmetic in every cell, a side of a 1024^2 level took 24 us.
//
// Walls are ghost values as in k_rbsweep.cu: x = b = 0 outside the domain, and K of the cell next
// to a wall is -K (Neumann: the face weight vanishes) or 3 K (Dirichlet: the half-cell weight).
// The ghosts are never relaxed. Periodic halos hold copies of the wrapped cells, relaxed like
// them. Arithmetic face mean only.
#pragma once
#include "fld_device.cuh"

namespace fld {

constexpr int T2_W = 64;

struct T2Args {
    const float *xin, *b, *K, *ec;     // xin null: the iterate starts from zero; ec: prolonged
    float *xout, *bc;                  // bc (nullable): the coarse right-hand side
    int sweeps, H, R;                  // R rows are loaded: tiles of (T2_W - 2H) x (R - 2H)
};

// halo of `sweeps` sweeps, with the residual after them
__host__ __device__ __forceinline__ int t2_halo(int sweeps, bool restricts) {
    return 2 * sweeps + (restricts ? 1 : 0);
}
// floats of shared memory of a tile: x, K, b, and a second x on odd periodic extents
__host__ __device__ constexpr int t2_floats(int R, bool odd) {
    return (odd ? 4 : 3) * T2_W * R;
}
__host__ __device__ __forceinline__ bool t2_odd(const Lvl& F) {
    return (F.bclo[0] == FLD_BC_PERIODIC && (F.n[0] & 1)) ||
           (F.bclo[1] == FLD_BC_PERIODIC && (F.n[1] & 1));
}

// cell index of coordinate g on an axis of extent n (periodic axes wrap), -1 / -2 for the
// ghost at the low / high wall, -3 farther out
__device__ __forceinline__ int t2_axis(int g, int n, bool per) {
    if (g >= 0 && g < n) return g;
    if (per) {
        g %= n;
        return g < 0 ? g + n : g;
    }
    return g == -1 ? -1 : g == n ? -2 : -3;
}

__device__ __forceinline__ float t2_ghost(int bc) { return bc == FLD_BC_DIRICHLET ? 3.f : -1.f; }

// The tile at (x0, y0) of level F by the block's NT threads; C the coarse level (read with ec or
// bc). Ends without a barrier after its last reads of shared memory.
template <int NT>
__device__ __forceinline__ void t2_tile(const Lvl& F, const Lvl& C, const T2Args& a, int x0, int y0,
                                        float* sm) {
    constexpr int W = T2_W, NW = NT / 32;
    const int nx = F.n[0], ny = F.n[1];
    const int R = a.R, H = a.H, N = W * R;
    const int tx = W - 2 * H, ty = R - 2 * H;
    float* X = sm;
    float* const K = sm + N;
    float* const B = sm + 2 * N;
    float* Y = sm + 3 * N;                                 // odd extents only
    const bool xper = F.bclo[0] == FLD_BC_PERIODIC, yper = F.bclo[1] == FLD_BC_PERIODIC;
    const bool odd = t2_odd(F);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;

    // ---- load, a warp a row, each lane its two columns
    {
        int gx[2];
        Interp ix[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            gx[e] = t2_axis(x0 - H + lane + 32 * e, nx, xper);
            if (a.ec) ix[e] = interp1(max(gx[e], 0), nx, C.n[0], F.bclo[0], F.bchi[0], F.pk);
        }
        for (int r = wid; r < R; r += NW) {
            const int gy = t2_axis(y0 - H + r, ny, yper);
            const bool row = gy >= 0, ghost = gy == -1 || gy == -2;
            const int base = (gy == -2 ? ny - 1 : max(gy, 0)) * nx;
            const float fy = ghost ? t2_ghost(gy == -1 ? F.bclo[1] : F.bchi[1]) : 1.f;
            Interp iy;
            if (a.ec) iy = interp1(max(gy, 0), ny, C.n[1], F.bclo[1], F.bchi[1], F.pk);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float xv = 0.f, kv = 0.f, bv = 0.f;
                if (gx[e] >= 0 && (row || ghost)) {
                    const int p = (int)fld_at((long long)base + gx[e], F.ncell);
                    kv = fy * a.K[p];
                    if (row) {
                        bv = a.b[p];
                        if (a.xin) xv = a.xin[p];
                        if (a.ec) {
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                const float* er = a.ec + (long long)iy.idx[q] * C.n[0];
                                xv += iy.wt[q] * (ix[e].wt[0] * er[ix[e].idx[0]] +
                                                  ix[e].wt[1] * er[ix[e].idx[1]]);
                            }
                        }
                    }
                } else if (row && (gx[e] == -1 || gx[e] == -2)) {
                    kv = t2_ghost(gx[e] == -1 ? F.bclo[0] : F.bchi[0]) *
                         a.K[base + (gx[e] == -1 ? 0 : nx - 1)];
                }
                const int o = r * W + lane + 32 * e;
                X[o] = xv;
                K[o] = kv;
                B[o] = bv;
            }
        }
    }
    __syncthreads();

    const float hx = 0.5f * F.wf[0], hy = 0.5f * F.wf[1];
    auto row_of = [&](int o, float& sw, float& acc) {
        const float kc = K[o];
        float f = (kc + K[o - 1]) * hx;
        sw = f;
        acc = f * X[o - 1];
        f = (kc + K[o + 1]) * hx;
        sw += f;
        acc = fmaf(f, X[o + 1], acc);
        f = (kc + K[o - W]) * hy;
        sw += f;
        acc = fmaf(f, X[o - W], acc);
        f = (kc + K[o + W]) * hy;
        sw += f;
        acc = fmaf(f, X[o + W], acc);
    };
    // ---- half sweeps, each on a region one cell smaller
    for (int s = 0; s < 2 * a.sweeps; ++s) {
        const int m = s + 1;                               // margin to the loaded region
        for (int r = m + wid; r < R - m; r += NW) {
            const int gy = y0 - H + r;
            if (odd) {                     // walls' rows and columns are copied as they are
                const int wy = t2_axis(gy, ny, yper);
                for (int c = lane; c < W; c += 32) {
                    const int wx = t2_axis(x0 - H + c, nx, xper);
                    const int o = r * W + c;
                    float v = X[o];
                    if (c >= m && c < W - m && wx >= 0 && wy >= 0 && ((wx + wy + s) & 1) == 0) {
                        float sw, acc;
                        row_of(o, sw, acc);
                        v = __fdividef(B[o] + acc, 1.f + sw);
                    }
                    Y[o] = v;
                }
                continue;
            }
            if (!yper && (gy < 0 || gy >= ny)) continue;
            // the cell of this colour in the lane's pair of columns
            const int c = 2 * lane + ((x0 - H + gy + s) & 1), gx = x0 - H + c;
            if (c < m || c >= W - m || (!xper && (gx < 0 || gx >= nx))) continue;
            float sw, acc;
            const int o = r * W + c;
            row_of(o, sw, acc);
            X[o] = __fdividef(B[o] + acc, 1.f + sw);
        }
        __syncthreads();
        if (odd) {
            float* const t = X;
            X = Y;
            Y = t;
        }
    }

    // ---- this tile's cells
    for (int r = wid; r < ty && y0 + r < ny; r += NW)
        for (int c = lane; c < tx && x0 + c < nx; c += 32)
            a.xout[fld_at((long long)(y0 + r) * nx + x0 + c, F.ncell)] = X[(r + H) * W + H + c];
    if (!a.bc) return;
    // ---- the mean of the children's residuals
    const int fx = C.n[0] < nx ? 2 : 1, fy = C.n[1] < ny ? 2 : 1;
    const int cw = tx / fx, ch = ty / fy, cx0 = x0 / fx, cy0 = y0 / fy;
    for (int r = wid; r < ch && cy0 + r < C.n[1]; r += NW)
        for (int c = lane; c < cw && cx0 + c < C.n[0]; c += 32) {
            float sum = 0.f;
            int cnt = 0;
            for (int q = 0; q < fy && (cy0 + r) * fy + q < ny; ++q)
                for (int p = 0; p < fx && (cx0 + c) * fx + p < nx; ++p) {
                    const int o = (r * fy + q + H) * W + H + c * fx + p;
                    float sw, acc;
                    row_of(o, sw, acc);
                    sum += B[o] - (1.f + sw) * X[o] + acc;
                    ++cnt;
                }
            a.bc[fld_at((long long)(cy0 + r) * C.n[0] + cx0 + c, C.ncell)] =
                sum * (cnt == 4 ? 0.25f : cnt == 2 ? 0.5f : 1.f);
        }
}

}  // namespace fld
