// Device parameters, cell routines and launchers of the one-dimensional radiation-MHD wave step.
#pragma once

#include <algorithm>

#include "fld_device.cuh"
#include "fld_line.cuh"

namespace fld {

// conservative <-> primitive (rho, v_x, v_y, v_z, B_y, B_z, p, E)
__device__ __forceinline__ void to_prim(const double* U, double Bx, double g, double* W) {
    const double rho = U[0];
    const double vx = U[1] / rho, vy = U[2] / rho, vz = U[3] / rho;
    W[0] = rho;
    W[1] = vx;
    W[2] = vy;
    W[3] = vz;
    W[4] = U[4];
    W[5] = U[5];
    W[6] = (g - 1.0) * (U[6] - 0.5 * rho * (vx * vx + vy * vy + vz * vz) -
                        0.5 * (Bx * Bx + U[4] * U[4] + U[5] * U[5]));
    W[7] = U[7];
}

__device__ __forceinline__ void to_cons(const double* W, double Bx, double g, double* U) {
    const double rho = W[0], vx = W[1], vy = W[2], vz = W[3];
    U[0] = rho;
    U[1] = rho * vx;
    U[2] = rho * vy;
    U[3] = rho * vz;
    U[4] = W[4];
    U[5] = W[5];
    U[6] = W[6] / (g - 1.0) + 0.5 * rho * (vx * vx + vy * vy + vz * vz) +
           0.5 * (Bx * Bx + W[4] * W[4] + W[5] * W[5]);
    U[7] = W[7];
}

// x-fluxes of the MHD equations and of E v_x (the advection term of the E equation)
__device__ __forceinline__ void phys_flux(const double* W, double Bx, double g, double* F) {
    const double rho = W[0], vx = W[1], vy = W[2], vz = W[3], By = W[4], Bz = W[5];
    const double p = W[6];
    const double B2 = Bx * Bx + By * By + Bz * Bz;
    const double pt = p + 0.5 * B2;
    const double e = p / (g - 1.0) + 0.5 * rho * (vx * vx + vy * vy + vz * vz) + 0.5 * B2;
    const double Bv = Bx * vx + By * vy + Bz * vz;
    F[0] = rho * vx;
    F[1] = rho * vx * vx + pt - Bx * Bx;
    F[2] = rho * vx * vy - Bx * By;
    F[3] = rho * vx * vz - Bx * Bz;
    F[4] = vx * By - Bx * vy;
    F[5] = vx * Bz - Bx * vz;
    F[6] = (e + pt) * vx - Bv * Bx;
    F[7] = W[7] * vx;
}

// fast magnetosonic speed from the gas sound speed sqrt(gamma p / rho)
__device__ __forceinline__ double fast_speed(const double* W, double Bx, double g) {
    const double rho = W[0];
    const double cs2 = g * W[6] / rho;
    const double va2 = (Bx * Bx + W[4] * W[4] + W[5] * W[5]) / rho;
    const double vax2 = Bx * Bx / rho;
    const double s = cs2 + va2;
    return sqrt(0.5 * (s + sqrt(fmax(s * s - 4.0 * cs2 * vax2, 0.0))));
}

// driving wave at cell centre x and time t, primitive variables
__device__ __forceinline__ void drive_prim(const Wave1dDev& P, double x, double t, double* W) {
    const double s = sin(P.k * x - P.omega * t);
#pragma unroll
    for (int v = 0; v < 8; ++v) W[v] = P.W0[v] + P.hat[v] * s;
}


// One explicit evaluation L(Uin) = -dF/dx + (0, f_r, 0, 0, 0, 0, v.f_r, -P:grad v) and the state
// formed from it: with ssp
//   Uout = a U0 + b (Uin + dt L),
// else (null operands have zero weight; the G's, [2][n], enter the gas energy and E)
//   Uout = U0 + dt (ca La + cb Lb + cn L) + dt (d2 G2 + d3 G3).
// Driven cells take the driving wave at t_out. Uout may alias U0.
struct W1Stage {
    const double *Uin, *U0, *La, *Lb, *G2, *G3;
    double *Uout, *Lout;           // Lout (nullable) receives L
    double a, b, ca, cb, cn, d2, d3, dt, t_in, t_out;
    int ssp, rad;                  // rad: with the coupling terms
    Opacity op;
    double c, E_right;
    int mode;                      // limiter
    unsigned* err;                 // domain flags of the coupling terms
    const unsigned* gate;          // nullable: Uout is left alone if the word is not zero
};

void launch_w1_advance(const Wave1dDev& P, const W1Stage& g, cudaStream_t s);
// the implicit stage of lines too long for one launch: primitive variables before the
// substep, its result into the state, the stage's increments
void launch_w1_prim(const Wave1dDev& P, const double* U, double* rho, double* T, double* T0,
                    double* E, cudaStream_t s);
void launch_w1_post(const Wave1dDev& P, double* U, const double* rho, const double* T0,
                    const double* T, const double* E, double t, cudaStream_t s);
void launch_w1_incr(const Wave1dDev& P, const double* Ua, const double* Ub, double inv_tau,
                    double* G, cudaStream_t s);
void launch_w1_speed(const Wave1dDev& P, const double* U, unsigned long long* out,
                     cudaStream_t s);

// The handle's side of it (fld_api.cu): whether its substep runs in one launch, the launch of
// stage `slot` (0 or 1) on the wave state, and the read-back of `slots` stages.
bool fld_line_wave_ok(const fld_handle* h);
fld_status fld_line_wave(fld_handle* h, const fld_consts* k, const fld_opacity* op, double tau,
                         const LineWave& w, const double* E_bc, int slot, cudaStream_t s);
fld_status fld_line_collect(fld_handle* h, int slots, fld_stats* st, cudaStream_t s);
const unsigned* fld_line_failed(fld_handle* h, int slot);   // device word of stage `slot`
unsigned* fld_handle_err(fld_handle* h);
bool fld_physics_ok(const fld_consts* k, const fld_opacity* op);
Opacity fld_to_opacity(const fld_opacity* op);

}  // namespace fld
