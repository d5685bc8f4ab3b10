// Kernels of the one-dimensional radiation-MHD wave step (Sect. 3 scheme, Sect. 4.3
// tests): primitive variables, WENO3 + HLL interface fluxes, the Runge-Kutta stage
// update with the explicit coupling sources, the exchange's energy feedback and the
// CFL signal speed. State arrays are variable-major [8][n]: rho, rho v_x, rho v_y,
// rho v_z, B_y, B_z, e (total gas energy), E; B_x is a constant.
#include <math_constants.h>

#include "fld_wave1d.cuh"

namespace fld {

namespace {

constexpr int W1_THREADS = 256;

// WENO3 states on both sides of the face between q0 and qp: two two-cell stencils per
// side with linear weights 1/3 and 2/3 and Jiang-Shu nonlinear weights; the smoothness
// indicators are divided by the largest square of the four cells (unit-free). The weights
// (1/3)/b0^2 and (2/3)/b1^2 are multiplied through by 3 b0^2 b1^2: three divisions in all.
__device__ __forceinline__ void weno3(double qm, double q0, double qp, double qpp, double& qL,
                                      double& qR) {
    const double eps = 1e-6;
    const double is = 1.0 / (fmax(fmax(qm * qm, q0 * q0), fmax(qp * qp, qpp * qpp)) + 1e-300);
    const double dm = q0 - qm, dc = qp - q0, dp = qpp - qp;
    const double bm = fma(dm * is, dm, eps), bc = fma(dc * is, dc, eps),
                 bp = fma(dp * is, dp, eps);
    const double wm = 2.0 * (bm * bm), wc = bc * bc, wp = 2.0 * (bp * bp);
    const double mid = fma(0.5, q0, 0.5 * qp);
    qL = fma(wc, fma(1.5, q0, -0.5 * qm), wm * mid) / (wc + wm);
    qR = fma(wc, fma(1.5, qp, -0.5 * qpp), wp * mid) / (wc + wp);
}

// primitive state of cell c: the driving wave left of the grid, zero gradient right of it
__device__ __forceinline__ void cell_prim(const Wave1dDev& P, const double* __restrict__ U,
                                          int c, double t, double* W) {
    if (c < 0) {
        drive_prim(P, (c + 0.5) * P.dx, t, W);
        return;
    }
    if (c >= P.n) c = P.n - 1;
    double u[8];
#pragma unroll
    for (int v = 0; v < 8; ++v) u[v] = U[(long long)v * P.n + c];
    to_prim(u, P.Bx, P.gamma, W);
}

__global__ void k_w1_prim(Wave1dDev P, const double* __restrict__ U, double* __restrict__ rho,
                          double* __restrict__ T, double* __restrict__ T0,
                          double* __restrict__ E) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.n) return;
    double W[8];
    cell_prim(P, U, i, 0.0, W);
    const double Tg = W[6] / (W[0] * P.R_gas);
    rho[i] = W[0];
    T[i] = T0[i] = Tg;
    E[i] = W[7];
}

// A whole explicit evaluation and the state formed from it, one launch in place of five
// (primitive variables, coupling terms, faces, right-hand side, combination). A line of a few
// thousand cells is bound by how few threads share its FP64 work, not by memory: one thread a
// face (7 blocks for 1600 cells) took 101 us for the faces alone. Here a block of four warps
// owns ADV_C cells and spreads the reconstruction over eight lanes a face, one a variable; 1600
// cells are 107 blocks. The values pass between the phases through shared memory.
constexpr int ADV_C = 15, ADV_F = ADV_C + 1, ADV_T = 8 * ADV_F, ADV_P = ADV_C + 4;

__global__ void __launch_bounds__(ADV_T)
k_w1_advance(Wave1dDev P, W1Stage g) {
    __shared__ double W[8][ADV_P];             // primitive variables of cells c0-2 .. c0+16
    __shared__ double Tg[ADV_P];
    __shared__ double Q[2][8][ADV_F];          // left and right states of the faces
    __shared__ double Uf[2][8][ADV_F], Ff[2][8][ADV_F], Sp[2][2][ADV_F];
    __shared__ double Fi[8][ADV_F];
    __shared__ double src[3][ADV_C];
    if (g.gate && *g.gate) return;
    const int c0 = blockIdx.x * ADV_C, tid = threadIdx.x;
    const long long n = P.n;
    if (tid < ADV_P) {
        double w[8];
        cell_prim(P, g.Uin, c0 - 2 + tid, g.t_in, w);
#pragma unroll
        for (int v = 0; v < 8; ++v) W[v][tid] = w[v];
        Tg[tid] = w[6] / (w[0] * P.R_gas);
    }
    __syncthreads();
    {
        const int f = tid >> 3, v = tid & 7;   // face f lies between cells c0+f-1 and c0+f
        double l, r;
        weno3(W[v][f], W[v][f + 1], W[v][f + 2], W[v][f + 3], l, r);
        Q[0][v][f] = l;
        Q[1][v][f] = r;
    }
    __syncthreads();
    if (tid < 2 * ADV_F) {
        // one side of a face: its conserved state, flux and signal speeds
        const int f = tid % ADV_F, sd = tid / ADV_F;
        double w[8], u[8], fl[8];
#pragma unroll
        for (int v = 0; v < 8; ++v) w[v] = Q[sd][v][f];
        to_cons(w, P.Bx, P.gamma, u);
        phys_flux(w, P.Bx, P.gamma, fl);
        const double cf = fast_speed(w, P.Bx, P.gamma);
#pragma unroll
        for (int v = 0; v < 8; ++v) {
            Uf[sd][v][f] = u[v];
            Ff[sd][v][f] = fl[v];
        }
        Sp[sd][0][f] = w[1] - cf;
        Sp[sd][1][f] = w[1] + cf;
    } else if (tid >= 64 && tid < 64 + ADV_C && c0 + tid - 64 < P.n) {
        // coupling terms of one cell (those of k_coupling on one axis): E's gradient with an
        // even mirror on the left and a Dirichlet face on the right, the velocity's with
        // even mirrors on both sides
        const int q = tid - 64, i = c0 + q;
        double fr = 0.0, vfr = 0.0, pt = 0.0;
        if (g.rad) {
            auto E = [&](int o) {
                const int c = i + o;
                if (c < 0) return W[7][-c - 1 - c0 + 2];
                if (c >= P.n) return 2.0 * g.E_right - W[7][2 * P.n - 1 - c - c0 + 2];
                return W[7][q + o + 2];
            };
            auto vx = [&](int o) {
                const int c = i + o;
                return W[1][(c < 0 ? -c - 1 : c >= P.n ? 2 * P.n - 1 - c : c) - c0 + 2];
            };
            const double ih = 1.0 / (12.0 * P.dx);
            const double Ec = E(0), r = W[0][q + 2];
            const double t = g.op.kind == FLD_OPACITY_CONST ? 1.0 : Tg[q + 2];
            bool ok = pos_finite(Ec) && pos_finite(r) && pos_finite(t);
            const double kap = ok ? opacity_eval(g.op, r, t) : 0.0;
            ok = ok && pos_finite(kap);
            if (ok) {
                const double gr = ((E(-2) - 8.0 * E(-1)) + 8.0 * E(1) - E(2)) * ih;
                const double dv = ((vx(-2) - 8.0 * vx(-1)) + 8.0 * vx(1) - vx(2)) * ih;
                const double R = sqrt(gr * gr) / (kap * r * Ec);
                const double lam = g.mode == FLD_LIMITER_LP
                                       ? (2.0 + R) / (6.0 + 3.0 * R + R * R)
                                       : g.mode == FLD_LIMITER_MINERBO ? minerbo_lambda(R)
                                                                       : 1.0 / 3.0;
                const double f = lam + lam * lam * R * R;
                fr = -lam * gr;
                vfr = vx(0) * fr;
                // P_xx = E f where the gradient has a direction, E (1 - f)/2 where it vanishes
                pt = (gr != 0.0 ? f : 0.5 * (1.0 - f)) * Ec * dv;
            } else {
                atomicOr(g.err, ERRBIT_DOMAIN);
            }
        }
        src[0][q] = fr;
        src[1][q] = vfr;
        src[2][q] = pt;
    }
    __syncthreads();
    {
        const int f = tid >> 3, v = tid & 7;
        const double SL = fmin(fmin(Sp[0][0][f], Sp[1][0][f]), 0.0);
        const double SR = fmax(fmax(Sp[0][1][f], Sp[1][1][f]), 0.0);
        Fi[v][f] = (SR * Ff[0][v][f] - SL * Ff[1][v][f] +
                    SL * SR * (Uf[1][v][f] - Uf[0][v][f])) / (SR - SL);
    }
    __syncthreads();
    const int v = tid / ADV_F, q = tid % ADV_F, i = c0 + q;    // consecutive cells a half-warp
    if (q >= ADV_C || i >= P.n) return;
    const long long at = v * n + i;
    double dU = -(Fi[v][q + 1] - Fi[v][q]) / P.dx;
    if (v == 1) dU += src[0][q];
    if (v == 6) dU += src[1][q];
    if (v == 7) dU -= src[2][q];
    if (g.Lout) g.Lout[at] = dU;
    double out;
    if (i < P.nd) {
        double w[8], u[8];
        drive_prim(P, (i + 0.5) * P.dx, g.t_out, w);
        to_cons(w, P.Bx, P.gamma, u);
        out = u[0];
#pragma unroll
        for (int e = 1; e < 8; ++e) out = v == e ? u[e] : out;
    } else if (g.ssp) {
        out = g.a * g.U0[at] + g.b * (g.Uin[at] + g.dt * dU);
    } else {
        double inc = 0.0;
        if (g.La) inc += g.ca * g.La[at];
        if (g.Lb) inc += g.cb * g.Lb[at];
        inc += g.cn * dU;
        if (v >= 6) {
            if (g.G2) inc += g.d2 * g.G2[(v - 6) * n + i];
            if (g.G3) inc += g.d3 * g.G3[(v - 6) * n + i];
        }
        out = g.U0[at] + g.dt * inc;
    }
    g.Uout[at] = out;
}

// the implicit increment of a stage: G = (Uafter - Ubefore) / tau for variables 6, 7
__global__ void k_w1_incr(Wave1dDev P, const double* __restrict__ Ua,
                          const double* __restrict__ Ub, double inv_tau, double* __restrict__ G) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.n) return;
    const long long n = P.n;
    G[i] = (Ua[6 * n + i] - Ub[6 * n + i]) * inv_tau;
    G[n + i] = (Ua[7 * n + i] - Ub[7 * n + i]) * inv_tau;
}

// after the FLD substep: e += rho R_gas (T' - T) / (gamma - 1), E = E'; driven cells reset
__global__ void k_w1_post(Wave1dDev P, double* __restrict__ U, const double* __restrict__ rho,
                          const double* __restrict__ T0, const double* __restrict__ T,
                          const double* __restrict__ E, double t) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.n) return;
    const long long n = P.n;
    if (i < P.nd) {
        double W[8], u[8];
        drive_prim(P, (i + 0.5) * P.dx, t, W);
        to_cons(W, P.Bx, P.gamma, u);
#pragma unroll
        for (int v = 0; v < 8; ++v) U[v * n + i] = u[v];
        return;
    }
    U[6 * n + i] += rho[i] * P.R_gas * (T[i] - T0[i]) / (P.gamma - 1.0);
    U[7 * n + i] = E[i];
}

// max over cells of |v_x| + c_f, as the bits of a non-negative double (integer order)
__global__ void k_w1_speed(Wave1dDev P, const double* __restrict__ U,
                           unsigned long long* __restrict__ out) {
    __shared__ double sh[W1_THREADS / 32];
    double s = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P.n; i += gridDim.x * blockDim.x) {
        double W[8];
        cell_prim(P, U, i, 0.0, W);
        const double c = fabs(W[1]) + fast_speed(W, P.Bx, P.gamma);
        // a cell with rho <= 0, p <= 0 or a non-finite speed makes the maximum +inf, which
        // the host reports as a domain error (fmax alone would drop a NaN)
        const bool ok = W[0] > 0.0 && W[6] > 0.0 && c < CUDART_INF;
        s = ok ? fmax(s, c) : CUDART_INF;
    }
    for (int o = 16; o > 0; o >>= 1) s = fmax(s, __shfl_xor_sync(0xffffffffu, s, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        s = threadIdx.x < W1_THREADS / 32 ? sh[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) s = fmax(s, __shfl_xor_sync(0xffffffffu, s, o));
        if (threadIdx.x == 0) atomicMax(out, (unsigned long long)__double_as_longlong(s));
    }
}

int blocks_for(long long n) { return (int)((n + W1_THREADS - 1) / W1_THREADS); }

}  // namespace

void launch_w1_prim(const Wave1dDev& P, const double* U, double* rho, double* T, double* T0,
                    double* E, cudaStream_t s) {
    k_w1_prim<<<blocks_for(P.n), W1_THREADS, 0, s>>>(P, U, rho, T, T0, E);
}

void launch_w1_advance(const Wave1dDev& P, const W1Stage& g, cudaStream_t s) {
    k_w1_advance<<<(P.n + ADV_C - 1) / ADV_C, ADV_T, 0, s>>>(P, g);
}

void launch_w1_post(const Wave1dDev& P, double* U, const double* rho, const double* T0,
                    const double* T, const double* E, double t, cudaStream_t s) {
    k_w1_post<<<blocks_for(P.n), W1_THREADS, 0, s>>>(P, U, rho, T0, T, E, t);
}

void launch_w1_incr(const Wave1dDev& P, const double* Ua, const double* Ub, double inv_tau,
                    double* G, cudaStream_t s) {
    k_w1_incr<<<blocks_for(P.n), W1_THREADS, 0, s>>>(P, Ua, Ub, inv_tau, G);
}

void launch_w1_speed(const Wave1dDev& P, const double* U, unsigned long long* out,
                     cudaStream_t s) {
    const int nb = std::min(blocks_for(P.n), num_sms() * 4);
    k_w1_speed<<<nb, W1_THREADS, 0, s>>>(P, U, out);
}

}  // namespace fld
