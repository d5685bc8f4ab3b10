// One side of a 2D FP32 multigrid level in one launch: a tile (tile2d.cuh) per block.
//
// 2D levels are small (a 1024^2 level is 4 MB a field, and stays in L2), so a V-cycle of half-sweep
// launches is bound by launches and by the latency of each: 30 of them took ~175 us at 1024^2,
// 5.8 us each, where the data of one passes through L2 in under 2 us. With two sweeps a tile
// relaxes 1.5 to 1.9 times its cells, and a V-cycle of three levels is five launches.
#include <algorithm>

#include "tile2d.cuh"

namespace fld {

namespace {

constexpr int T2_NT = 512;

__global__ void __launch_bounds__(T2_NT) k_tile2d(Lvl F, Lvl C, T2Args a) {
    after_previous();
    extern __shared__ float t2[];
    t2_tile<T2_NT>(F, C, a, blockIdx.x * (T2_W - 2 * a.H), blockIdx.y * (a.R - 2 * a.H), t2);
}

}  // namespace

bool tile2d_ok(const Lvl& L, int sweeps) {
    return L.ndim == 2 && !L.fm && sweeps <= TILE2D_SWEEPS && L.n[1] <= 65535;
}

void prepare_tile2d() {
    cudaFuncSetAttribute(k_tile2d, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sizeof(float) * t2_floats(48, true));
}

void launch_tile2d(const Lvl& F, const Lvl& C, const float* xin, float* xout, const float* b,
                   const float* K, const float* ec, float* bc, int sweeps, cudaStream_t s) {
    T2Args a;
    a.xin = xin;
    a.xout = xout;
    a.b = b;
    a.K = K;
    a.ec = ec;
    a.bc = bc;
    a.sweeps = sweeps;
    a.H = t2_halo(sweeps, bc != nullptr);
    // 48 rows where the tiles fill the GPU, 32 below: more blocks, each done sooner
    const int tx = T2_W - 2 * a.H;
    const bool big = (long long)F.n[0] * F.n[1] >= (long long)tx * (48 - 2 * a.H) * num_sms();
    a.R = big ? 48 : 32;
    const int ty = a.R - 2 * a.H;
    const dim3 grid((F.n[0] + tx - 1) / tx, (F.n[1] + ty - 1) / ty);
    launch_chained(true, k_tile2d, grid, T2_NT, sizeof(float) * t2_floats(a.R, t2_odd(F)), s, F, C,
                   a);
}

}  // namespace fld
