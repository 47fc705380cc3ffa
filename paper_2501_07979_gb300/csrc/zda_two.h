// Two time steps per launch on (phi, z) tiles streamed along r (zda_two.cu).
#pragma once
#include "zda_internal.h"

namespace zda {

constexpr int TWO_THREADS = 384;       // most threads of a block

// How a zone is cut: tiles_j x tiles_k tiles, each streamed over `ranges` ranges of radii.
struct TwoPlan {
    int tiles_j = 0, tiles_k = 0, ranges = 0;   // 0: the zone cannot take this step
    int full = 0;                      // a tile holds every phi row (no halo rows; the wedge wraps inside it)
    int nrow = 0, npair = 0;           // rows and z-pairs of a tile with its halo: one thread each
    int nzq = 0;                       // most z-pairs of a tile that lie in the z-PML
    size_t smem = 0;
    double cost = 0;                   // estimate of a launch's time, in units of about 1.8 ns
    int threads() const { return (nrow * npair + 31) / 32 * 32; }
};

// CPML auxiliaries, first the H side, then the E side: z slabs, r slabs
enum { PS_HR_Z, PS_HP_Z, PS_ER_Z, PS_EP_Z, PS_HP_R, PS_HZ_R, PS_EP_R, PS_EZ_R, PS_N };

struct TwoParams {
    StepParams p;                      // tables, density, source, DFT history (its fields and psi are not used)
    const float2 *iE[3], *iH[3], *iP[PS_N];     // state before step n
    float2 *oE[3], *oH[3], *oP[PS_N];           // state after step n + 1 (other buffers)
    int tiles_k, tiles_j, i_range, full, nrow, npair, nzq;
};

bool two_applies(const StepParams &p);
// rows: most phi rows per tile (8 or 16), ranges: radius ranges (0: chosen here)
TwoPlan two_plan(const StepParams &p, int rows, int ranges, int sms, size_t smem_limit);
// p.src_rad: adjoint sources of steps n and n + 1, [2][2][n_r]
cudaError_t launch_two(const TwoPlan &pl, const TwoParams &q, int n, cudaStream_t s);

}  // namespace zda
