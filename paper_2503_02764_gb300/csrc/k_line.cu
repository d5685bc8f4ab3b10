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
// cluster's FP64 issue (13 steps of 17 instructions a row on 8 SMs, ~60 us) costs as much as
// their launches do.
//
// The system and the method are those of k_tridiag.cu (parallel cyclic reduction,
// Sherman-Morrison for periodic lines, FP64 refinement steps until the residual meets tol), with
// rows scaled to a unit diagonal: a step then takes one reciprocal (an FP32 seed and two
// Newton-Raphson steps) in place of two divisions, 14 FP64 instructions a row, or 17 with the
// second right-hand side, in place of about 40.
#include <cooperative_groups.h>

#include "fld_device.cuh"
#include "fld_line.cuh"
#include "fld_wave1d.cuh"

namespace cg = cooperative_groups;

namespace fld {

namespace {

constexpr int LINE_CS = 8;          // blocks of the cluster (the portable maximum)
constexpr int LINE_T = 256;
constexpr int LINE_ARRAYS = 13;     // K, b, x, r, kappa rho, two sets of a, c, d, e

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
    double* A[2] = {arr + 5 * m, arr + 6 * m};
    double* Cc[2] = {arr + 7 * m, arr + 8 * m};
    double* Dd[2] = {arr + 9 * m, arr + 10 * m};
    double* Ee[2] = {arr + 11 * m, arr + 12 * m};
    const int first = rank << lg;
    const int mine = max(0, min(m, n - first));      // rows of this block
    const bool per = g.L.bclo[0] == FLD_BC_PERIODIC;
    // a value of row i, wherever it lives
    auto at = [&](double* p, int i) -> double {
        return cl.map_shared_rank(p, i >> lg)[i & (m - 1)];
    };
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
        for (int q = threadIdx.x; q < mine; q += LINE_T) {
            const int i = first + q;
            const double Ki = K[q];
            double wl = 0.0, wr = 0.0, dg = 1.0, e = 0.0;
            if (i > 0) wl = fmean(Ki, at(K, i - 1), g.L.fm);
            else if (per) wl = fmean(Ki, at(K, n - 1), g.L.fm);
            else if (g.L.bclo[0] == FLD_BC_DIRICHLET) dg = fma(2.0, Ki, dg);
            if (i < n - 1) wr = fmean(Ki, at(K, i + 1), g.L.fm);
            else if (per) wr = fmean(Ki, at(K, 0), g.L.fm);
            else if (g.L.bchi[0] == FLD_BC_DIRICHLET) dg = fma(2.0, Ki, dg);
            dg += wl + wr;
            double ai = -wl, ci = -wr;
            if (per && i == 0) {                   // the corners go into u v^T
                e = -dg;                           // u_0 = gamma
                ai = 0.0;
                dg += dg;                          // dg - gamma
            }
            if (per && i == n - 1) {
                e = ci;
                dg = fma(ratio, wr, dg);           // dg - a_0 c_{n-1} / gamma
                ci = 0.0;
            }
            const double inv = 1.0 / dg;
            A[0][q] = ai * inv;
            Cc[0][q] = ci * inv;
            Dd[0][q] = f[q] * inv;
            if (per) Ee[0][q] = e * inv;
        }
        int cur = 0;
        cl.sync();
        for (int st = 1; st < n; st *= 2) {
            const int nxt = cur ^ 1;
            for (int q = threadIdx.x; q < mine; q += LINE_T) {
                const int i = first + q, im = i - st, ip = i + st;
                const double a = A[cur][q], c = Cc[cur][q];
                double am = 0.0, cm = 0.0, dm = 0.0, em = 0.0, ap = 0.0, cp = 0.0, dp = 0.0,
                       ep = 0.0;
                if (im >= 0) {
                    am = at(A[cur], im);
                    cm = at(Cc[cur], im);
                    dm = at(Dd[cur], im);
                    if (per) em = at(Ee[cur], im);
                }
                if (ip < n) {
                    ap = at(A[cur], ip);
                    cp = at(Cc[cur], ip);
                    dp = at(Dd[cur], ip);
                    if (per) ep = at(Ee[cur], ip);
                }
                // the scaled rows are diagonally dominant: 1 - a cm - c ap > 0, at most 1
                const double piv = fma(-c, ap, fma(-a, cm, 1.0));
                const double r = in_f32_range(piv) && piv > 0.0 ? rcp_nr(piv) : 1.0 / piv;
                A[nxt][q] = -a * am * r;
                Cc[nxt][q] = -c * cp * r;
                Dd[nxt][q] = fma(-c, dp, fma(-a, dm, Dd[cur][q])) * r;
                if (per) Ee[nxt][q] = fma(-c, ep, fma(-a, em, Ee[cur][q])) * r;
            }
            cur = nxt;
            cl.sync();
        }
        double s = 0.0;
        if (per) {
            // v = (1, 0, .., a_0/gamma); a_0 / gamma = wc / dg_0 > 0
            const double y0 = at(Dd[cur], 0), yn = at(Dd[cur], n - 1);
            const double z0 = at(Ee[cur], 0), zn = at(Ee[cur], n - 1);
            s = fma(ratio, yn, y0) / (1.0 + fma(ratio, zn, z0));
        }
        for (int q = threadIdx.x; q < mine; q += LINE_T) {
            const double y = per ? fma(-s, Ee[cur][q], Dd[cur][q]) : Dd[cur][q];
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
