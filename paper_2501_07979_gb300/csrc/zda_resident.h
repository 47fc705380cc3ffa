// Whole time loop of a small zone in one launch, its state held on the SMs (zda_resident.cu).
#pragma once
#include "zda_internal.h"

namespace zda {

constexpr int RES_THREADS = 512;       // most threads of a brick's block
constexpr int RES_THREADS_1 = 320;     // ... with one own cell per thread (and so more registers each)
constexpr int RES_MAX_CELLS = 4;       // most own cells per thread

// A zone cut into gi x gj x gk bricks, one thread block each.
struct ResidentPlan {
    int gi = 0, gj = 0, gk = 0;        // bricks per direction; 0: the zone does not fit
    int threads = 0, per_thread = 0;   // block size, own cells per thread
    size_t smem = 0;                   // dynamic shared memory of a block
    int blocks() const { return gi * gj * gk; }
};

struct ResidentParams {
    StepParams p;
    int gi, gj, gk;
    int nkz_h, nkz_e, nir_h, nir_e;    // largest z- and r-slab extents of any brick (H range, own cells)
    int n_recv;                        // capacity of the halo list
    int n0, n1, n_steps;               // steps [n0, n1) of a run of n_steps
    uint4 *mail;                       // halo packets [2][3][cells]
    int *err;                          // error word: a bounded wait gave up
    int wait_limit, inject_timeout;
};

ResidentPlan resident_plan(const StepParams &p, int sms, size_t smem_limit);
size_t resident_mail_bytes(int nr, int nphi, int nz);
cudaError_t launch_resident(const ResidentPlan &pl, const StepParams &p, int n0, int n1, int n_steps, void *mail,
                            int *err, int wait_limit, int inject_timeout, cudaStream_t s);

}  // namespace zda
