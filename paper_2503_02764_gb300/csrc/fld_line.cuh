// The 1D substep and direct solve in one launch (k_line.cu).
#pragma once
#include "fld_device.cuh"

namespace fld {

constexpr int LINE_CELLS = 8192;      // cells; longer lines run k_tridiag.cu's launches

struct LineOut {                    // written by the kernel, read back with the scalars
    double rel;                     // final relative residual
    double hist[64];                // relative residual before and after each solve
    int cyc;                        // solves (0: a cell failed the domain check)
};

struct LineArgs {
    Lvl L;
    BcOff bo;
    Opacity op;
    const double *rho, *D, *Ebc;    // D: the caller's coefficient (solve alone)
    double *T, *E;
    double inv12h, kscale, c, dtc, a_r, cv, tol, one;   // one = 1.0
    int mode, max_cycles;           // mode: the limiter
};

bool line_ok(const Lvl& L);
void prepare_line();
void launch_line(const LineArgs& g, bool step, LineOut* out, unsigned* err, cudaStream_t s);

}  // namespace fld
