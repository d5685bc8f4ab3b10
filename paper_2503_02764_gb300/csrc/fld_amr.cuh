// Declarations shared by the composite-grid solve's kernels (k_amr.cu) and its host side
// (fld_amr_api.cu).
#pragma once
#include <algorithm>

#include "fld_internal.cuh"

namespace fld {

// Geometry of a coarse block with one box refined by 2 (axes beyond nd have n = 1).
struct AmrGeom {
    int nd;
    int nc[3];              // coarse cells per axis
    int nf[3];              // fine cells per axis: 2 (hi - lo)
    int lo[3], hi[3];       // the box in coarse indices (hi exclusive)
    int bclo[3], bchi[3];
    double H[3];            // coarse cell sizes
    double dt;
    long long bcoff[6];     // offset of each Dirichlet face block in E_bc (-1: none)
};

void launch_amr_setup(const AmrGeom& G, const double* Dc, const double* Df, const double* Ec,
                      const double* Ef, const double* Ebc, double* bc, double* bf, double* DH,
                      cudaStream_t s);
// Rows of one grid, formed once per solve: face conductances per axis (extent + 1 along it)
// and inverse diagonals.
struct AmrRows {
    double* w[3];
    double* inv;
};
// x: readable values of both grids (their faces are walked, the values not used)
void launch_amr_rows(const AmrGeom& G, const AmrRows& Rc, const AmrRows& Rf, const double* Dc,
                     const double* Df, const double* xc, const double* xf, cudaStream_t s);
void launch_amr_smooth(const AmrGeom& G, const AmrRows& Rc, const AmrRows& Rf, int phase,
                       const double* bc, const double* bf, double* xc, double* xf,
                       cudaStream_t s);
int launch_amr_resid(const AmrGeom& G, const AmrRows& Rc, const AmrRows& Rf, const double* bc,
                     const double* bf, const double* xc, const double* xf, double* rc, double* rf,
                     double* partials, int nblocks, cudaStream_t s);
void launch_amr_average(const AmrGeom& G, const double* vf, double* vc, cudaStream_t s);
void launch_amr_correct(const AmrGeom& G, const double* e, double* xc, double* xf,
                        cudaStream_t s);

// The block's multigrid as the coarse correction (fld_api.cu): the operator of D over dt set up
// once per solve, then `cycles` V-cycles on A e = r from e = 0, without a read-back. `scale`, a
// power of two, brings r to order one, where the FP32 V-cycles of the mixed modes hold it.
fld_status fld_correction_setup(fld_handle* h, double dt, const double* D, const double* r,
                                cudaStream_t s);
fld_status fld_correction(fld_handle* h, const double* r, double scale, double* e, int cycles,
                          cudaStream_t s);

}  // namespace fld
