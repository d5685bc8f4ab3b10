// The 1D substep (limiter -> direct solve -> exchange) and the 1D direct solve alone, in one
// launch of one thread-block cluster for lines of up to LINE_CELLS cells.
//
// The separate launches (k_limiter, k_prep_level0, the norms, a dozen of k_pcr_step, k_exchange)
// and their four read-backs took 208 us for 256 cells, nearly all of it launch and
// synchronisation latency. One block would hold such a line, but one SM issues only 4 G FP64
// instructions a second, so the rows are spread over the eight SMs of a cluster: rows and
// right-hand sides stay in shared memory, neighbours are read from the blocks that own them
// (distributed shared memory), and a cluster barrier (~0.3 us) takes the place of each
// launch. Longer lines keep the launches over the whole GPU (k_tridiag.cu): at 8192 cells the
// cluster's FP64 issue (13 steps of 14 instructions a row on 8 SMs, ~60 us) costs as much as
// their launches do.
//
// The system and the method are those of k_tridiag.cu (parallel cyclic reduction,
// Sherman-Morrison for periodic lines, FP64 refinement steps until the residual meets tol). A
// row keeps the reciprocal of its diagonal (an FP32 seed and two Newton-Raphson steps), so that a
// step divides by its neighbours' diagonals with two multiplications: 14 FP64 instructions a
// row, or 16 with the second right-hand side, in place of about 40.
//
// In place of the diagonal b a row keeps its excess g = b - a - c over the couplings a, c >= 0
// to its neighbours. Eliminating both gives
//   a' = k1 a_-, c' = k2 c_+, g' = g + k1 g_- + k2 g_+, d' = d + k1 d_- + k2 d_+,
// with k1 = a / b_-, k2 = c / b_+: sums and products of positive numbers, in which nothing
// cancels however large dt D / h^2 is. Restated on the CPU against 113-bit solutions (lines of 32
// to 4096 cells, walls), the largest relative error is 1.0e-15 at K = 30, 300 and 30000; with
// the diagonal itself (k_tridiag.cu) 4e-15, 2e-14 and 4e-13, with rows scaled to a unit
// diagonal 5e-15, 2e-14 and 6e-13.
#include <cooperative_groups.h>

#include "fld_device.cuh"
#include "fld_line.cuh"
#include "fld_wave1d.cuh"

namespace cg = cooperative_groups;

namespace fld {

namespace {

constexpr int LINE_CS = 8;          // blocks of the cluster (the portable maximum)
constexpr int LINE_T = 256;
constexpr int LINE_ARRAYS = 17;     // K, b, x, r, kappa rho, two sets of a, c, g, 1/b, d, e

struct LineShared {
    double red[32];
    double part[2];
};

template <int KIND>
__global__ void __cluster_dims__(LINE_CS, 1, 1) __launch_bounds__(LINE_T)
k_line(LineArgs g, int lg, LineOut* out, unsigned* err) {
    constexpr bool STEP = KIND != LINE_SOLVE;
    extern __shared__ double arr[];
    __shared__ LineShared sh;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int m = 1 << lg, n = g.L.n[0];
    double* const K = arr;
    double* const B = arr + m;
    double* const X = arr + 2 * m;
    double* const Rr = arr + 3 * m;
    double* const KR = arr + 4 * m;
    const int first = rank << lg;
    const int mine = max(0, min(m, n - first));      // rows of this block
    const bool per = g.L.bclo[0] == FLD_BC_PERIODIC;
    // row i of an array, and its value, wherever it lives
    auto row = [&](double* p, int i) -> const double* {
        return cl.map_shared_rank(p, i >> lg) + (i & (m - 1));
    };
    auto at = [&](double* p, int i) -> double { return *row(p, i); };
    // the reduction's set of arrays `cur`: a, c, g, 1/b, d, e, m doubles each
    auto set = [&](int cur) { return arr + (5 + 6 * cur) * m; };
    // sums over the cluster: fixed trees in the blocks, then the blocks in rank order
    auto csum = [&](double v) -> double {
        v = block_sum(v, sh.red);
        if (threadIdx.x == 0) sh.part[0] = v;
        cl.sync();
        double t = 0.0;
        for (int r = 0; r < LINE_CS; ++r) t += cl.map_shared_rank(sh.part, r)[0];
        cl.sync();
        return t;
    };

    // ---- D (the limiter's or the caller's), K, b
    double bad = 0.0, b2 = 0.0;
    if (threadIdx.x == 0 && rank == 0 && *err) bad = 1.0;      // flagged by an earlier call
    const double ih[3] = {g.inv12h, 0.0, 0.0};
    for (int q = threadIdx.x; q < mine; q += LINE_T) {
        const int i = first + q;
        double Dp, lm;
        if (KIND == LINE_WAVE) {          // the gas temperature of the conserved state
            double u[8], W[8];
            for (int v = 0; v < 8; ++v) u[v] = g.w.Uin[(long long)v * n + i];
            to_prim(u, g.w.P.Bx, g.w.P.gamma, W);
            g.T[i] = W[6] / (W[0] * g.w.P.R_gas);
        }
        if (STEP) {
            double kr = 0.0;
            if (!limiter_cell(g.L, ih, g.E, g.rho, g.T, g.Ebc, g.bo, g.op, g.c, g.mode, i, 0, 0, i,
                              Dp, lm, &kr, false, g.one)) {
                bad = 1.0;
                Dp = 0.0;
            }
            KR[q] = kr;
        } else {
            Dp = g.D[i];
        }
        if (!pos_finite(Dp)) bad = 1.0;
        const double Kp = g.kscale * Dp;
        double bp = g.E[i];
        if (g.Ebc) {
            if (i == 0 && g.L.bclo[0] == FLD_BC_DIRICHLET) bp = fma(2.0 * Kp, g.Ebc[g.bo.off[0]], bp);
            if (i == n - 1 && g.L.bchi[0] == FLD_BC_DIRICHLET)
                bp = fma(2.0 * Kp, g.Ebc[g.bo.off[1]], bp);
        }
        K[q] = Kp;
        B[q] = bp;
        X[q] = g.E[i];
        b2 = fma(bp, bp, b2);
    }
    if (csum(bad) > 0.0) {
        if (rank == 0 && threadIdx.x == 0) {
            atomicOr(err, ERRBIT_DOMAIN);
            out->cyc = 0;
            out->rel = 0.0;
            out->failed = 1u;
        }
        return;
    }
    const double bnorm = sqrt(csum(b2));

    // r = b - A x into Rr, and its relative norm
    auto residual = [&]() -> double {
        double r2 = 0.0;
        for (int q = threadIdx.x; q < mine; q += LINE_T) {
            const int i = first + q;
            const double Ki = K[q], xi = X[q];
            const int il = i > 0 ? i - 1 : (per ? n - 1 : -1);
            const int ir = i < n - 1 ? i + 1 : (per ? 0 : -1);
            double r = fma(xi, -g.one, B[q]);
            if (il >= 0) r = fma(fmean(Ki, at(K, il), g.L.fm), fma(xi, -g.one, at(X, il)), r);
            else if (g.L.bclo[0] == FLD_BC_DIRICHLET) r = fma(-2.0 * Ki, xi, r);
            if (ir >= 0) r = fma(fmean(Ki, at(K, ir), g.L.fm), fma(xi, -g.one, at(X, ir)), r);
            else if (g.L.bchi[0] == FLD_BC_DIRICHLET) r = fma(-2.0 * Ki, xi, r);
            Rr[q] = r;
            r2 = fma(r, r, r2);
        }
        r2 = csum(r2);
        return bnorm > 0.0 ? sqrt(r2) / bnorm : 0.0;
    };

    // y = A^-1 f for the right-hand side f of this block's rows, left in X (add: added to it)
    auto solve = [&](const double* f, bool add) {
        double ratio = 0.0;                        // a_0 / gamma (periodic)
        if (per) {
            const double wc = fmean(at(K, 0), at(K, n - 1), g.L.fm);
            ratio = wc / (1.0 + wc + fmean(at(K, 0), at(K, 1), g.L.fm));
        }
        auto inverse = [](double b) { return in_f32_range(b) ? rcp_nr(b) : 1.0 / b; };
        for (int q = threadIdx.x; q < mine; q += LINE_T) {
            const int i = first + q;
            const double Ki = K[q];
            double wl = 0.0, wr = 0.0, ex = 1.0, e = 0.0;
            if (i > 0) wl = fmean(Ki, at(K, i - 1), g.L.fm);
            else if (!per && g.L.bclo[0] == FLD_BC_DIRICHLET) ex = fma(2.0, Ki, ex);
            if (i < n - 1) wr = fmean(Ki, at(K, i + 1), g.L.fm);
            else if (!per && g.L.bchi[0] == FLD_BC_DIRICHLET) ex = fma(2.0, Ki, ex);
            if (per && i == 0) {                   // the corners go into u v^T
                const double wc = fmean(Ki, at(K, n - 1), g.L.fm);
                e = -(1.0 + wc + wr);              // u_0 = gamma = -b_0
                ex = fma(2.0, 1.0 + wc, wr);       // 2 b_0 - wr
            }
            if (per && i == n - 1) {
                const double wc = fmean(Ki, at(K, 0), g.L.fm);
                e = -wc;
                ex = fma(ratio, wc, 1.0 + wc);     // b - wl - a_0 c_{n-1} / gamma
            }
            double* const w = set(0) + q;
            w[0] = wl;
            w[m] = wr;
            w[2 * m] = ex;
            w[3 * m] = inverse(ex + (wl + wr));
            w[4 * m] = f[q];
            if (per) w[5 * m] = e;
        }
        int cur = 0;
        cl.sync();
        for (int st = 1; st < n; st *= 2) {
            double* const S = set(cur);
            double* const N = set(cur ^ 1);
            for (int q = threadIdx.x; q < mine; q += LINE_T) {
                const int i = first + q, im = i - st, ip = i + st;
                double an = 0.0, cn = 0.0, gn = S[2 * m + q], dn = S[4 * m + q];
                double en = per ? S[5 * m + q] : 0.0;
                if (im >= 0) {
                    const double* const w = row(S, im);
                    const double k = S[q] * w[3 * m];
                    an = k * w[0];
                    gn = fma(k, w[2 * m], gn);
                    dn = fma(k, w[4 * m], dn);
                    if (per) en = fma(k, w[5 * m], en);
                }
                if (ip < n) {
                    const double* const w = row(S, ip);
                    const double k = S[m + q] * w[3 * m];
                    cn = k * w[m];
                    gn = fma(k, w[2 * m], gn);
                    dn = fma(k, w[4 * m], dn);
                    if (per) en = fma(k, w[5 * m], en);
                }
                N[q] = an;
                N[m + q] = cn;
                N[2 * m + q] = gn;
                N[3 * m + q] = inverse(gn + (an + cn));
                N[4 * m + q] = dn;
                if (per) N[5 * m + q] = en;
            }
            cur ^= 1;
            cl.sync();
        }
        // no row has neighbours left: a = c = 0, and the diagonal is g
        double* const S = set(cur);
        double s = 0.0;
        if (per) {
            // v = (1, 0, .., a_0/gamma); a_0 / gamma = wc / b_0 > 0
            const double* const w0 = row(S, 0);
            const double* const wn = row(S, n - 1);
            const double g0 = w0[2 * m], gn = wn[2 * m], d0 = w0[4 * m], dn = ratio * wn[4 * m];
            const double e0 = w0[5 * m], en = ratio * wn[5 * m];
            // (y_0 + ratio y_n) / (1 + z_0 + ratio z_n) with y = d / g, z = e / g, in one division
            // (256 periodic cells: 37.8 us in the kernel with five, 35.8)
            if (in_f32_range(g0) && in_f32_range(gn))
                s = fma(dn, g0, d0 * gn) / fma(g0, gn, fma(en, g0, e0 * gn));
            else
                s = (dn / gn + d0 / g0) / (1.0 + (en / gn + e0 / g0));
        }
        for (int q = threadIdx.x; q < mine; q += LINE_T) {
            const double d = S[4 * m + q];
            const double y = (per ? fma(-s, S[5 * m + q], d) : d) / S[2 * m + q];
            X[q] = add ? X[q] + y : y;
        }
        cl.sync();
    };

    double rel = residual();                       // of E^n, as the V-cycle path reports it
    if (rank == 0 && threadIdx.x == 0) out->hist[0] = rel;
    solve(B, false);
    int cyc = 1;
    for (;;) {
        rel = residual();
        if (rank == 0 && threadIdx.x == 0 && cyc < 64) out->hist[cyc] = rel;
        if (!(rel > g.tol) || cyc >= g.max_cycles || !isfinite(rel)) break;
        solve(Rr, true);
        ++cyc;
    }
    if (rank == 0 && threadIdx.x == 0) {
        out->cyc = cyc;
        out->rel = rel;
        out->failed = 0u;
    }
    if (KIND == LINE_WAVE) {
        // nothing is written unless every cell of the line passes
        double fail = isfinite(rel) ? 0.0 : 1.0;
        for (int q = threadIdx.x; q < mine; q += LINE_T) {
            const int i = first + q;
            const double r = g.rho[i], kr = KR[q];
            double t = g.T[i], er = X[q];
            if (pos_finite(kr) && pos_finite(r) && pos_finite(t) && pos_finite(er))
                exchange_cell_kr(r, kr, t, er, g.dtc, g.a_r, g.cv, g.one);
            else
                fail = 1.0;
            KR[q] = t - g.T[i];
            X[q] = er;
        }
        if (csum(fail) > 0.0) {
            // the flag stops the step's next stage, which would read this one's outputs
            if (rank == 0 && threadIdx.x == 0) {
                atomicOr(err, ERRBIT_DOMAIN);
                out->failed = 1u;
            }
            return;
        }
        const Wave1dDev& P = g.w.P;
        for (int q = threadIdx.x; q < mine; q += LINE_T) {
            const int i = first + q;
            double u[8];
            for (int v = 0; v < 8; ++v) u[v] = g.w.Uin[(long long)v * n + i];
            const double e0 = u[6], E0 = u[7];
            u[6] += u[0] * P.R_gas * KR[q] / (P.gamma - 1.0);
            u[7] = X[q];
            if (i < P.nd) {
                double W[8];
                drive_prim(P, (i + 0.5) * P.dx, g.w.t_drive, W);
                to_cons(W, P.Bx, P.gamma, u);
            }
            for (int v = 0; v < 8; ++v) g.w.Uout[(long long)v * n + i] = u[v];
            if (g.w.G) {
                g.w.G[i] = (u[6] - e0) * g.w.inv_tau;
                g.w.G[n + i] = (u[7] - E0) * g.w.inv_tau;
            }
        }
        return;                                    // the sum above was the last remote read
    }
    const bool ex = STEP && isfinite(rel);         // a diverged solve ends before the exchange
    for (int q = threadIdx.x; q < mine; q += LINE_T) {
        const int i = first + q;
        double er = X[q];
        if (ex) {
            const double r = g.rho[i], kr = KR[q];
            double t = g.T[i];
            if (pos_finite(kr) && pos_finite(r) && pos_finite(t) && pos_finite(er)) {
                exchange_cell_kr(r, kr, t, er, g.dtc, g.a_r, g.cv, g.one);
                g.T[i] = t;
            } else {
                atomicOr(err, ERRBIT_DOMAIN);
            }
        }
        g.E[i] = er;
    }
    cl.sync();                                     // no block leaves while its rows are read
}

int line_lg(int n) {
    int lg = 2;
    while ((LINE_CS << lg) < n) ++lg;
    return lg;
}

size_t line_smem(int lg) { return sizeof(double) * LINE_ARRAYS * ((size_t)1 << lg); }

}  // namespace

bool line_ok(const Lvl& L) { return L.ndim == 1 && L.n[0] <= LINE_CELLS; }

void prepare_line() {
    const int most = (int)line_smem(line_lg(LINE_CELLS));
    cudaFuncSetAttribute(k_line<LINE_SOLVE>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    cudaFuncSetAttribute(k_line<LINE_STEP>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    cudaFuncSetAttribute(k_line<LINE_WAVE>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
}

void launch_line(const LineArgs& g, int kind, LineOut* out, unsigned* err, cudaStream_t s) {
    const int lg = line_lg(g.L.n[0]);
    const size_t sm = line_smem(lg);
    if (kind == LINE_STEP) k_line<LINE_STEP><<<LINE_CS, LINE_T, sm, s>>>(g, lg, out, err);
    else if (kind == LINE_WAVE) k_line<LINE_WAVE><<<LINE_CS, LINE_T, sm, s>>>(g, lg, out, err);
    else k_line<LINE_SOLVE><<<LINE_CS, LINE_T, sm, s>>>(g, lg, out, err);
}

}  // namespace fld
