// Batched substep: per-problem descriptors and the persistent kernel's launcher.
#pragma once
#include "fld_internal.cuh"
#include "tile2d.cuh"

namespace fld {

constexpr int BMAXL = 16;   // multigrid levels per batched problem

// Device-resident descriptor of one batched problem.
struct BProb {
    Lvl lv[BMAXL];          // level geometry (level 0 = the problem's grid)
    long long o32[BMAXL];   // offset (floats) of level l's FP32 arrays x, b, K, t in the
                            // problem's FP32 workspace (x at o32, b at +n, K +2n, t +3n)
    double kdown[BMAXL];    // K_{l+1} = mean(K_l children) * kdown[l]
    int nlev;
    double h[3];            // cell sizes (x, y, z)
    long long cell_off;     // first cell of the problem in the concatenated fields
    long long ebc_off;      // first Dirichlet face value in the concatenated faces (-1: none)
    long long bc_off[6];    // Dirichlet face blocks within the problem's faces (-1: none)
    long long ws_d;         // offset (doubles) of the problem's FP64 workspace: D, then
                            // the FP64 refinement's x, b and K (4 n doubles)
    long long ws_f;         // offset (floats) of the problem's FP32 workspace
};

// Per-call data of one problem (uploaded each step).
struct BDyn {
    double dt;              // time step
    Opacity op;             // opacity law
};

struct BatchParams {
    double c, a_r, cv;      // speed of light, radiation constant, R_gas/(gamma - 1)
    double tol;
    int max_cycles, nu1, nu2, coarse_sweeps, limiter, inner;
    int tiles;              // 1: a problem of the batch runs its V-cycles on tiles
    int fp64;               // 1: FP64 refinement, limiter and exchange; 0: double-FP32
};

struct BatchStat {
    int cycles;
    double rel_resid;       // final relative residual (-1 on a domain error)
    double rel_resid0;      // before the first cycle
};

// Rows that a block of nt threads loads a tile of.
__host__ __device__ constexpr int batch_tile_rows(int nt) { return nt >= 512 ? 48 : 32; }
// Whether a problem's V-cycles run on tiles (tile2d.cuh) or as half sweeps, for groups of cs
// blocks of nt threads (times of 600 equal problems on tiles / as half sweeps, MIXED, V(1,1)).
//  - Blocks of 1024 threads, one an SM: half sweeps. A tile has too few cells for them, and no
//    other block fills the time of its barriers and loads (512 problems of 32 to 512 cells a
//    side: 45.2 / 40.7 ms).
//  - A cluster: tiles at every size, a barrier of the cluster in place of three (two blocks of
//    512, 16^2: 1.9 / 2.7 ms; 97^2: 6.7 / 8.3; 256^2: 24.9 / 30.3).
//  - A single block waits for little in a half sweep of a small problem, and the cells that tiles
//    load twice, or beyond the last row or column, are what counts. 512 threads: 32^2
//    1.39 / 1.36 ms, 64^2 (loaded 2.4 times) 2.66 / 2.28, 128^2 (1.8 times) 7.1 / 6.4, 112^2 (1.3)
//    5.0 / 5.2, 160^2 (1.4) 9.3 / 9.9, 256^2 23.3 / 27.6; more sweeps a load weigh against more
//    loads (V(2,2): 128^2, twice, 5.6 / 5.8). 256 threads have half as many loads in flight:
//    128^2 (1.9 times) 8.7 / 8.8, 192^2 (1.7) 18.0 / 20.8, V(2,2) 112^2 (2.6) 5.7 / 6.5. Below 8192
//    cells neither gains 4 %.
//  - Odd periodic extents, whose half sweeps go through a second copy of the tile: from 65536 cells
//    on (97^2 5.4 / 4.8 ms, 193^2 16.8 / 16.8).
__host__ __device__ inline bool batch_tiled(const Lvl& L, int nt, int cs, int nu1, int nu2) {
    if (nt >= 1024 || L.ndim != 2 || nu1 > TILE2D_SWEEPS || nu2 > TILE2D_SWEEPS) return false;
    if (cs > 1 || L.ncell >= 65536) return true;
    if (L.ncell < 8192 || t2_odd(L)) return false;
    const int H = t2_halo(nu1, true), tx = T2_W - 2 * H, ty = batch_tile_rows(nt) - 2 * H;
    const long long ntx = (L.n[0] + tx - 1) / tx, nty = (L.n[1] + ty - 1) / ty;
    const long long loaded = ntx * T2_W * (L.n[1] + 2 * H * nty);
    const int nu = nu1 > nu2 ? nu1 : nu2;
    return 20 * loaded <= (20 + (nt >= 512 ? 12 : 17) * nu) * L.ncell;
}

int batch_threads_supported(int nt);
int batch_cluster_supported(int cs);
// groups (clusters of cs blocks of nt threads) that can be resident at once
int batch_max_groups(int nt, int cs, const BatchParams& prm);
// the same, and the launch, for one block size, with or without tiles (batch_step.cuh)
template <int NT, bool TILED>
int batch_groups(int cs);
template <int NT, bool TILED>
void batch_launch(int cs, int ngroups, const BProb* probs, const BDyn* dyn, const int* order,
                  int nprob, int* queue, const BatchParams& prm, const double* rho, double* T,
                  double* E, const double* Ebc, double* wsd, float* wsf, BatchStat* stats,
                  unsigned* err, cudaStream_t s);
void launch_batch_step(int nt, int cs, int ngroups, const BProb* probs, const BDyn* dyn,
                       const int* order, int nprob, int* queue, const BatchParams& prm,
                       const double* rho, double* T, double* E, const double* Ebc, double* wsd,
                       float* wsf, BatchStat* stats, unsigned* err, cudaStream_t s);

}  // namespace fld
