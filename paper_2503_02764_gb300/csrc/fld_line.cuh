// The 1D substep and direct solve in one launch (k_line.cu).
#pragma once
#include "fld_device.cuh"

namespace fld {

constexpr int LINE_CELLS = 8192;      // cells; longer lines run k_tridiag.cu's launches

struct LineOut {                    // written by the kernel, read back with the scalars
    double rel;                     // final relative residual
    double hist[64];                // relative residual before and after each solve
    int cyc;                        // solves (0: a cell failed the domain check)
    unsigned failed;                // LINE_WAVE: not zero if nothing was written
};

struct Wave1dDev {
    int n, nd;                  // cells, driven cells at the left end
    double dx, gamma, Bx, R_gas;
    double W0[8], hat[8];       // driving wave W0 + hat sin(k x - omega t), primitive
    double k, omega;
};

// the wave step's implicit stage on its conserved state: U_out = U_in with the substep's change of
// gas energy and E, driven cells at t_drive, G (nullable) the increments of both over tau
struct LineWave {
    Wave1dDev P;
    const double* Uin;
    double *Uout, *T, *G;           // T: n doubles of scratch
    double inv_tau, t_drive;
};

struct LineArgs {
    Lvl L;
    BcOff bo;
    Opacity op;
    const double *rho, *D, *Ebc;    // D: the caller's coefficient (solve alone)
    double *T, *E;
    double inv12h, kscale, c, dtc, a_r, cv, tol, one;   // one = 1.0
    int mode, max_cycles;           // mode: the limiter
    LineWave w;
};

bool line_ok(const Lvl& L);
void prepare_line();
// LINE_SOLVE: E <- A^-1 (E + walls); LINE_STEP: the whole substep on (T, E); LINE_WAVE: the
// wave step's implicit stage
enum { LINE_SOLVE, LINE_STEP, LINE_WAVE };
void launch_line(const LineArgs& g, int kind, LineOut* out, unsigned* err, cudaStream_t s);

}  // namespace fld
