// Pointwise kernels of the FLD substep: the gas-radiation exchange quartic and the
// flux limiter (Levermore-Pomraning, 4th-order 5-point gradient).
#include <algorithm>

#include "fld_device.cuh"

namespace fld {

// ----------------------------------------------------------------- exchange
// Backward Euler on de/dt = +qdot, dE/dt = -qdot with qdot = c kappa rho (E - a_r T^4)
// (Eqs. heating, qdot). Eliminating E' and multiplying by 1 + chi, chi = dt c kappa rho, leaves,
// per cell,
//   f(T) = alpha T + beta T^4 - q = 0,  alpha = rho c_v (1 + chi), beta = a_r chi,
//   q = alpha T^n + chi E,
// increasing and convex for T > 0 with f(0) < 0: one positive root, bounded above by
// min(q/alpha, (q/beta)^(1/4)), from where Newton decreases monotonically to it.
//
// FP64 arithmetic is the scarce resource on this GPU, so the root is found in two
// stages: Newton in FP32 on a scaled form of the quartic (all quantities O(1)), then
// one FP64 Newton step, whose residual f(T) is evaluated in FP64 and whose derivative
// only needs FP32 accuracy (the step is ~1e-7 T, so a 1e-7 relative error in it leaves
// ~1e-14 T). Cells whose coefficients fall outside the FP32 range take a plain FP64
// Newton iteration instead.

// kr (nullable): kappa rho of every cell, frozen at the step's start by the limiter of the
// same substep; without it kappa is evaluated from (rho, T). DF as for k_limiter.
template <bool DF>
__global__ void __launch_bounds__(256, 5) k_exchange(long long n, const double* __restrict__ rho, double* __restrict__ T,
                           double* __restrict__ E, const double* __restrict__ kr, Opacity op,
                           double dtc, double a_r, double cv, int use_df, DfConst K,
                           unsigned* err, double one) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const double r = rho[i];
        double t = T[i], er = E[i];
        const double kri = kr ? kr[i] : 0.0;
        if (kr && !pos_finite(kri)) {
            atomicOr(err, ERRBIT_DOMAIN);
            continue;
        }
        if (DF && use_df && exchange_cell_df(r, t, er, op, K, kri)) {
            T[i] = t;
            E[i] = er;
            continue;
        }
        t = T[i];
        er = E[i];
        if (kr) {
            if (!(pos_finite(r) && pos_finite(t) && pos_finite(er))) {
                atomicOr(err, ERRBIT_DOMAIN);
                continue;
            }
            exchange_cell_kr(r, kri, t, er, dtc, a_r, cv, one);
        } else if (!exchange_cell(r, t, er, op, dtc, a_r, cv)) {
            atomicOr(err, ERRBIT_DOMAIN);
            continue;
        }
        T[i] = t;
        E[i] = er;
    }
}

DfConst make_dfconst(double c, double kappa0, double dtc, double a_r, double cv) {
    DfConst K;
    split_host(c, K.c_h, K.c_l);
    split_host(kappa0, K.kap_h, K.kap_l);
    split_host(dtc, K.dtc_h, K.dtc_l);
    split_host(a_r, K.ar_h, K.ar_l);
    split_host(cv, K.cv_h, K.cv_l);
    return K;
}

void launch_exchange(long long n, const double* rho, double* T, double* E, Opacity op,
                     double dtc, double a_r, double cv, int use_df, unsigned* err, cudaStream_t s,
                     const double* kr) {
    if (n <= 0) return;
    const int block = 256;
    long long nb = (n + block - 1) / block;
    if (nb > num_sms() * 32) nb = num_sms() * 32;
    const DfConst K = make_dfconst(0.0, op.kappa0, dtc, a_r, cv);
    if (use_df)
        k_exchange<true><<<(int)nb, block, 0, s>>>(n, rho, T, E, kr, op, dtc, a_r, cv, use_df, K,
                                                   err, 1.0);
    else
        k_exchange<false><<<(int)nb, block, 0, s>>>(n, rho, T, E, kr, op, dtc, a_r, cv, use_df, K,
                                                    err, 1.0);
}

// ----------------------------------------------------------------- limiter
// E split into FP32 (hi, lo) pairs, once per cell, for the double-FP32 limiter's gradient
__global__ void k_split_df(long long n, const double* __restrict__ v, float* __restrict__ hi,
                           float* __restrict__ lo) {
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n;
         p += (long long)gridDim.x * blockDim.x) {
        const df d = df_from_double_i(v[p]);
        hi[p] = d.hi;
        lo[p] = d.lo;
    }
}

// The FP64 routine of the cells that the double-FP32 one declines, out of line: its registers
// would cost the double-FP32 kernel its fifth block per SM.
static __device__ __noinline__ bool limiter_cell_64(const Lvl& L, const double* ih, const double* E,
                                                    const double* rho, const double* T,
                                                    const double* Ebc, const BcOff& bo,
                                                    const Opacity& op, double c, int mode, int i,
                                                    int j, int k, long long p, double& D,
                                                    double& lm, double* kr) {
    return limiter_cell(L, ih, E, rho, T, Ebc, bo, op, c, mode, i, j, k, p, D, lm, kr);
}

struct Df3 {             // 1/(12 h_d) as pairs, split once on the host
    df v[3];
};

// kr (nullable): receives kappa rho of every cell, for the exchange of the same substep.
// DF: the double-FP32 cell routine first (FP64 for the cells it declines); the FP64-only
// instantiation carries none of its registers.
template <bool DF>
__global__ void __launch_bounds__(256, DF ? 5 : 4) k_limiter(Lvl L, double3 inv12h, Df3 inv12hd, const double* __restrict__ E,
                          const double* __restrict__ rho, const double* __restrict__ T,
                          const double* __restrict__ Ebc, BcOff bo, Opacity op, double c,
                          int mode, int use_df, DfConst K, const float* __restrict__ Eh,
                          const float* __restrict__ El, double* __restrict__ D,
                          double* __restrict__ lam, double* __restrict__ kr, unsigned* err,
                          double one) {
    const double ih[3] = {inv12h.x, inv12h.y, inv12h.z};
    const df ihd[3] = {inv12hd.v[0], inv12hd.v[1], inv12hd.v[2]};
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L.n[0]) return;
    for (int k = blockIdx.z; k < L.n[2]; k += gridDim.z)
        for (int j = blockIdx.y * blockDim.y + threadIdx.y; j < L.n[1];
             j += gridDim.y * blockDim.y) {
            const long long p = ((long long)k * L.n[1] + j) * L.n[0] + i;
            double Dv, lm, kv;
            if (DF && use_df && limiter_cell_df(L, ih, E, rho, T, Ebc, bo, op, K, mode, i, j, k, p, Dv, lm,
                                          Eh, El, ihd, kr ? &kv : nullptr)) {
                D[p] = Dv;
                if (lam) lam[p] = lm;
                if (kr) kr[p] = kv;
                continue;
            }
            if (!(DF ? limiter_cell_64(L, ih, E, rho, T, Ebc, bo, op, c, mode, i, j, k, p, Dv, lm,
                                       &kv)
                     : limiter_cell(L, ih, E, rho, T, Ebc, bo, op, c, mode, i, j, k, p, Dv, lm,
                                    kr ? &kv : nullptr, lam != nullptr, one))) {
                atomicOr(err, ERRBIT_DOMAIN);
                continue;
            }
            D[p] = Dv;
            if (lam) lam[p] = lm;
            if (kr) kr[p] = kv;
        }
}

// ----------------------------------------------------------------- coupling terms
// v_-2, v_-1, v_+1, v_+2 along axis d: periodic wrap, an even mirror at walls.
__device__ __forceinline__ void fetch_v(const Lvl& L, const double* __restrict__ v, int c, int d,
                                        int p, double w[4]) {
    const int n = L.n[d], st = d == 0 ? 1 : d == 1 ? L.n[0] : L.n[0] * L.n[1];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        int m = c + (q < 2 ? q - 2 : q - 1);
        if (m < 0) m = L.bclo[d] == FLD_BC_PERIODIC ? m + n : -m - 1;
        else if (m >= n) m = L.bchi[d] == FLD_BC_PERIODIC ? m - n : 2 * n - 1 - m;
        w[q] = v[p + (m - c) * st];
    }
}

// Explicit coupling terms of one cell, in FP64 from the limiter's gradient: F = -D grad E,
// f_r = -lambda grad E, f = lambda + lambda^2 R^2, and with v: v . f_r and
// P : grad v, P = E ((1 - f) I + (3f - 1) n n) / 2, n = grad E / |grad E|, contracted as
//   E ((1 - f)/2 div v + (3f - 1)/(2 g^2) sum_ij g_i g_j d_j v_i).
// FP64 issue bounds it (88 % of the pipe with IEEE divisions and roots and the twelve
// differences in FP64, 166 instructions a cell): lambda / a is one fix_div as in the limiter,
// lambda R = g (lambda / a), and the differences run in fixed point (fix64.cuh).
__global__ void __launch_bounds__(256, 3)
k_coupling(Lvl L, double3 inv12h, const double* __restrict__ E,
           const double* __restrict__ rho, const double* __restrict__ T,
           const double* __restrict__ Ebc, BcOff bo, Opacity op, double c,
           int mode, const double* __restrict__ v, double* __restrict__ F,
           double* __restrict__ fr, double* __restrict__ fe,
           double* __restrict__ vfr, double* __restrict__ pt, unsigned* err, double one) {
    const double ih[3] = {inv12h.x, inv12h.y, inv12h.z};
    const long long nc = L.ncell;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L.n[0]) return;
    for (int k = blockIdx.z; k < L.n[2]; k += gridDim.z)
        for (int j = blockIdx.y * blockDim.y + threadIdx.y; j < L.n[1];
             j += gridDim.y * blockDim.y) {
            const int p = (k * L.n[1] + j) * L.n[0] + i;
            const double Ec = E[p], r = rho[p];
            const double t = op.kind == FLD_OPACITY_CONST ? 1.0 : T[p];
            double kr;
            if (!(pos_finite(Ec) && pos_finite(r) && pos_finite(t)) ||
                !kapparho<true>(op, r, t, kr)) {
                atomicOr(err, ERRBIT_DOMAIN);
                continue;
            }
            double g[3] = {0.0, 0.0, 0.0};
            double g2 = 0.0;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                if (d >= L.ndim) break;
                double w[4];
                fetch_axis(L, E, Ebc, bo, i, j, k, d, p, w);
                g[d] = fix_stencil(w[0], w[1], w[2], w[3]) * ih[d];
                g2 = fma(g[d], g[d], g2);
            }
            const double a = kr * Ec;
            double lam, lr, D, gn, q;          // lr = lambda R
            bool far = false;                  // |grad E|^2 near the ends of the FP64 range
            if (mode != FLD_LIMITER_DIFFUSION && limiter_core<true>(a, g2, mode, one, true, gn, q, lam)) {
                lr = gn * q;
                D = c * Ec * q;
            } else {
                gn = sqrt(g2);
                far = abs((__double2hiint(g2) >> 20) - 1023) > 300 && gn > 0.0;
                const double R = gn / a;
                lam = mode == FLD_LIMITER_LP        ? (2.0 + R) / (6.0 + 3.0 * R + R * R)
                      : mode == FLD_LIMITER_MINERBO ? minerbo_lambda(R)
                                                    : 1.0 / 3.0;
                lr = lam * R;
                D = c * lam / kr;
            }
            const double f = fma(lr, lr, lam);
            double vf = 0.0;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                if (d >= L.ndim) break;
                const double frd = -lam * g[d];
                if (F) F[d * nc + p] = -D * g[d];
                if (fr) fr[d * nc + p] = frd;
                if (v) vf = fma(v[d * nc + p], frd, vf);
            }
            if (fe) fe[p] = f;
            if (v && vfr) vfr[p] = vf;
            if (v && pt) {
                // n n has no scale: where 1 / g^2, or g^2 times grad v, could leave the FP64 range,
                // g is brought to order one first (at 2^-514, for instance, g^2 is subnormal). The
                // empty statement keeps the FP64 instructions in their branch: they would be
                // executed speculatively by every cell.
                if (far) {
                    asm volatile("");
                    const int e = (__double2hiint(g2) >> 20) - 1023;
                    const double sc =
                        __hiloint2double((1023 + max(-511, min(-(e / 2), 511))) << 20, 0);
                    g2 = 0.0;
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        g[d] *= sc;
                        g2 = fma(g[d], g[d], g2);
                    }
                }
                double gh[3], div = 0.0, S = 0.0;
                const int cc[3] = {i, j, k};
#pragma unroll
                for (int d = 0; d < 3; ++d) gh[d] = d < L.ndim ? g[d] * ih[d] : 0.0;
#pragma unroll
                for (int a1 = 0; a1 < 3; ++a1) {             // velocity component
                    if (a1 >= L.ndim) break;
                    const double* vi = v + a1 * nc;
                    double gv = 0.0;
#pragma unroll
                    for (int a2 = 0; a2 < 3; ++a2) {         // derivative axis
                        if (a2 >= L.ndim) break;
                        double w[4];
                        fetch_v(L, vi, cc[a2], a2, p, w);
                        const double s = fix_stencil(w[0], w[1], w[2], w[3]);
                        gv = fma(gh[a2], s, gv);
                        if (a1 == a2) div = fma(ih[a2], s, div);
                    }
                    S = fma(g[a1], gv, S);
                }
                double acc = 0.5 * fma(f, -one, 1.0) * div;
                if (gn > 0.0) {
                    const double bq = fma(1.5, f, -0.5);
                    acc = fma(div_ok(1.0, g2) ? bq * fix_div(1.0, g2) : bq / g2, S, acc);
                }
                pt[p] = Ec * acc;
            }
        }
}

// blocks of 32 x 8 cells, or of a line's cells in a row
static dim3 cell_block(const Lvl& L) { return L.n[1] > 1 ? dim3(32, 8) : dim3(256, 1); }
// and a thread's planes: up to four, as long as six blocks an SM remain (the launch constants are
// loaded once a thread; the double-FP32 limiter of 256^3 takes 801 us with one plane a thread)
static dim3 cell_grid(const Lvl& L, dim3 blk) {
    const int gx = (L.n[0] + blk.x - 1) / blk.x;
    const int gy = std::min<int>((L.n[1] + blk.y - 1) / blk.y, 65535);
    int gz = std::min(L.n[2], 65535);
    while (gz > 1 && 4LL * gz > L.n[2] && (long long)gx * gy * (gz / 2) >= 6LL * num_sms())
        gz = (gz + 1) / 2;
    return dim3(gx, gy, gz);
}

void launch_coupling(const Lvl& L, const double* h, const double* E, const double* rho,
                     const double* T, const double* E_bc, const long long* bc_off, Opacity op,
                     double c, int mode, const double* v, double* F, double* fr, double* fe,
                     double* vfr, double* pt, unsigned* err, cudaStream_t s) {
    BcOff bo;
    for (int q = 0; q < 6; ++q) bo.off[q] = bc_off[q];
    const double3 ih = make_double3(1.0 / (12.0 * h[0]), L.ndim > 1 ? 1.0 / (12.0 * h[1]) : 0.0,
                                    L.ndim > 2 ? 1.0 / (12.0 * h[2]) : 0.0);
    const dim3 blk = cell_block(L);
    k_coupling<<<cell_grid(L, blk), blk, 0, s>>>(L, ih, E, rho, T, E_bc, bo, op, c, mode, v, F,
                                                 fr, fe, vfr, pt, err, 1.0);
}

void launch_split_df(long long n, const double* v, float* hi, float* lo, cudaStream_t s) {
    const long long nb = std::min<long long>((n + 255) / 256, num_sms() * 32);
    k_split_df<<<(int)nb, 256, 0, s>>>(n, v, hi, lo);
}

void launch_limiter(const Lvl& L, const double* h, const double* E, const double* rho,
                    const double* T, const double* E_bc, const long long* bc_off, Opacity op,
                    double c, int mode, int use_df, double* D, double* lam, unsigned* err,
                    cudaStream_t s, float* Eh, float* El, double* kr) {
    BcOff bo;
    for (int q = 0; q < 6; ++q) bo.off[q] = bc_off[q];
    double3 ih = make_double3(1.0 / (12.0 * h[0]), L.ndim > 1 ? 1.0 / (12.0 * h[1]) : 0.0,
                              L.ndim > 2 ? 1.0 / (12.0 * h[2]) : 0.0);
    const dim3 block = cell_block(L), nb = cell_grid(L, block);
    const DfConst K = make_dfconst(c, op.kappa0, 0.0, 0.0, 0.0);
    Df3 ihd;
    split_host(ih.x, ihd.v[0].hi, ihd.v[0].lo);
    split_host(ih.y, ihd.v[1].hi, ihd.v[1].lo);
    split_host(ih.z, ihd.v[2].hi, ihd.v[2].lo);
    if (!(use_df && mode != FLD_LIMITER_DIFFUSION)) Eh = El = nullptr;
    if (use_df)
        k_limiter<true><<<nb, block, 0, s>>>(L, ih, ihd, E, rho, T, E_bc, bo, op, c, mode, use_df, K,
                                             Eh, El, D, lam, kr, err, 1.0);
    else
        k_limiter<false><<<nb, block, 0, s>>>(L, ih, ihd, E, rho, T, E_bc, bo, op, c, mode, use_df, K,
                                              Eh, El, D, lam, kr, err, 1.0);
}

}  // namespace fld
