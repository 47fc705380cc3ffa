// Resident time loop (sm_103a): every step of a small zone's run in one launch.
//
// What it is for: on a zone of up to about three hundred thousand cells the two
// or three launches of a split step cost 10-17 us, its arithmetic 1 us or so.
// Here the zone is cut into bricks of cells, one thread block per brick and
// SM, and a brick's state stays on its SM for the whole run: E and H in shared
// memory (with one cell per thread in registers as well), CPML auxiliaries in
// shared memory, each cell's dt / eps in its thread's registers.  Per step
// only the faces of E cross between bricks.  Measured per step (a topology
// optimisation iteration's time over its steps): 24 x 8 x 40 cells 10.4 us by
// launches, 3.0 here; 248 x 1 x 160 (axis zone) 16.7 and 2.3; 48 x 48 x 64
// 11.0 and 4.6; 64 x 50 x 64 17.5 and 8.5; 60 x 40 x 100 19.4 and 12.0.  So it
// is taken wherever the zone fits (512 threads x 4 own cells per brick and its
// state in the brick's shared memory), but where the launches of a step are
// wanted or others share the GPU: a kernel chosen explicitly, event timing, the
// decay probe, a lens, a stream capture, runs of one step, and forward runs
// whose final fields may have decayed.
//
// What bounds it: small bricks the exchange (1.4 us of 2.3-3: a store to L2
// and a load from it, across both dies); large ones shared-memory bandwidth,
// 29 eight-byte accesses per cell and step.
//
// One exchange per step: a brick also carries the H cells one layer below it
// in each direction and updates them itself from the halo of E, so only
// E^{n+1} has to cross, once, between the E and the next H update.  A copy
// sees its owner's arithmetic on its owner's values and stays equal to it bit
// by bit; the copy of the wedge's last row below its first is kept without the
// Bloch phase for that reason (with the phase in, its rounding left a static
// charge along the seam: field error 7e-6 instead of 1.4e-6 after 1000 steps).
//
// The launch is cooperative (all bricks resident).  Every boundary value
// travels as one 16-byte packet {re, tag, im, tag} through L2, tag = the step:
// the reader polls the packet itself, so no fence or flag is on the path.
// Packets are double-buffered by step parity; neighbours read from each other,
// so a packet is only overwritten after its reader has sent the step in
// between.  Waits are bounded; a brick that gives up sets the error word and
// leaves, and the caller repeats the run by the split step.  (As one thread-block cluster, with the halo read from the
// neighbours' shared memory, a step of the 24 x 8 x 40 zone took 4.1 us: the
// cluster barriers cost as much as the packets and 16 SMs hold too few warps.)
//
// Complex values are updated with the packed FP32 instructions (two lanes per
// instruction).  Each update adds its whole curl to the field in one rounding,
// as the split step does.  The running DFTs keep the split step's time-blocked
// form: E at the DFT sites goes to the history buffer, and every DFT_BLOCK
// steps each brick folds its own sites into the accumulators while its halo is
// under way.
#include "zda_resident.h"

#include <algorithm>
#include <cmath>

namespace zda {

namespace {

typedef unsigned long long u64;

__device__ __forceinline__ u64 bits(float2 a) { return *reinterpret_cast<u64 *>(&a); }
__device__ __forceinline__ float2 pair(u64 a) { return *reinterpret_cast<float2 *>(&a); }
__device__ __forceinline__ float2 both(float s) { return make_float2(s, s); }
__device__ __forceinline__ float2 padd(float2 a, float2 b)
{
    u64 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(bits(a)), "l"(bits(b)));
    return pair(r);
}
__device__ __forceinline__ float2 pmul(float2 a, float2 b)
{
    u64 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(bits(a)), "l"(bits(b)));
    return pair(r);
}
__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c)
{
    u64 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(bits(a)), "l"(bits(b)), "l"(bits(c)));
    return pair(r);
}
__device__ __forceinline__ float2 psub(float2 a, float2 b) { return pfma(b, make_float2(-1.f, -1.f), a); }

// Bloch phase times a value with its roundings spelled out: the owner of a wrapped row and the brick that
// carries a copy of it must get the same bits.
__device__ __forceinline__ float2 turn(float2 ph, float2 v)
{
    return make_float2(__fmaf_rn(ph.x, v.x, -__fmul_rn(ph.y, v.y)), __fmaf_rn(ph.x, v.y, __fmul_rn(ph.y, v.x)));
}

__device__ __forceinline__ void send_packet(uint4 *at, float2 v, uint32_t tag)
{
    const u64 lo = (u64)__float_as_uint(v.x) | ((u64)tag << 32), hi = (u64)__float_as_uint(v.y) | ((u64)tag << 32);
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(at), "l"(lo), "l"(hi) : "memory");
}
__device__ __forceinline__ void read_packet(const uint4 *at, u64 &lo, u64 &hi)
{
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(lo), "=l"(hi) : "l"(at) : "memory");
}
__device__ __forceinline__ u64 now_ns()
{
    u64 t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// Per-radius table row, dt and 1/dphi (or m on the axis zone) folded in where the updates want them.
constexpr int ITAB = 16;
constexpr int SRC_BLOCK = 32;          // steps of the source's time table held at once
enum { T_HA, T_HB, T_HC, T_EA, T_EB, T_EC, T_BRN, T_CRN, T_BRH, T_CRH, T_IRN, T_IRH, T_BMN, T_CMN, T_BMH, T_CMH };

// Shared-memory layout of a brick, the same on the host (its size) and on the
// device; extents are the largest of any brick.
struct ResLayout {
    int ei, ej, ek;                    // own cells
    int XI, XJ, XK, NX;                // with the halo on both sides (none in phi on the axis zone)
    int cellsH;                        // H range: the own cells and the layers below them
    int E, H, pzH, prH, pmH, pzE, prE, pmE, src, kt, ph, tw, recv, itab, ztab, ctl;   // byte offsets
    int bytes;
};

__host__ __device__ __forceinline__ int brick_lo(int b, int n, int g) { return (int)((long long)b * n / g); }

__host__ __device__ __forceinline__ ResLayout res_layout(int nr, int nphi, int nz, int gi, int gj, int gk, int bor, int rm,
                                                         int nq, int nkz_h, int nkz_e, int nir_h, int nir_e, int n_recv)
{
    ResLayout L;
    L.ei = (nr + gi - 1) / gi;
    L.ej = (nphi + gj - 1) / gj;
    L.ek = (nz + gk - 1) / gk;
    L.XI = L.ei + 2;
    L.XJ = L.ej + (bor ? 0 : 2);
    L.XK = L.ek + 2;
    L.NX = L.XI * L.XJ * L.XK;
    const int eh = L.ei + (gi > 1), jh = L.ej + (gj > 1), kh = L.ek + (gk > 1);
    L.cellsH = eh * jh * kh;
    int o = 0;
    L.E = o; o += 3 * L.NX * 8;
    L.H = o; o += 3 * L.NX * 8;
    L.pzH = o; o += 2 * eh * jh * nkz_h * 8;
    L.prH = o; o += 2 * nir_h * jh * kh * 8;
    L.pmH = o; o += rm ? 2 * nir_h * jh * kh * 8 : 0;
    L.pzE = o; o += 2 * L.ei * L.ej * nkz_e * 8;
    L.prE = o; o += 2 * nir_e * L.ej * L.ek * 8;
    L.pmE = o; o += rm ? 2 * nir_e * L.ej * L.ek * 8 : 0;
    L.src = o; o += 2 * 2 * (L.ei + 1) * 8;
    L.kt = o; o += 2 * SRC_BLOCK * nq * 8;
    L.ph = o; o += 2 * L.ej * 8;
    o = (o + 15) & ~15;
    L.tw = o; o += DFT_BLOCK * nq * 16;
    L.recv = o; o += n_recv * 8;
    o = (o + 15) & ~15;
    L.itab = o; o += (L.ei + 1) * ITAB * 4;
    L.ztab = o; o += (L.ek + 1) * 16;
    L.ctl = o; o += 16;
    L.bytes = o;
    return L;
}

// Which components of E a brick needs at a halo cell in direction (di, dj, dk)
// (bit c: component c): what its H cells and the H layer below it read.
__host__ __device__ __forceinline__ int halo_need(int di, int dj, int dk)
{
    const int key = (di + 1) * 9 + (dj + 1) * 3 + (dk + 1);
    switch (key) {
    case 0 * 9 + 1 * 3 + 1:                            // low faces: the redundant H layer
    case 1 * 9 + 0 * 3 + 1:
    case 1 * 9 + 1 * 3 + 0: return 7;
    case 2 * 9 + 1 * 3 + 1: return 6;                  // high r: E_phi, E_z
    case 1 * 9 + 2 * 3 + 1: return 5;                  // high phi: E_r, E_z
    case 1 * 9 + 1 * 3 + 2: return 3;                  // high z: E_r, E_phi
    case 0 * 9 + 1 * 3 + 2:                            // edges next to a low face
    case 0 * 9 + 2 * 3 + 1: return 1;
    case 1 * 9 + 0 * 3 + 2:
    case 2 * 9 + 0 * 3 + 1: return 2;
    case 1 * 9 + 2 * 3 + 0:
    case 2 * 9 + 1 * 3 + 0: return 4;
    default: return 0;
    }
}

// Bits of a cell's flags; above them the row of the per-radius table and the own phi row (10 bits each).
enum { F_ACT = 1, F_TURN_H = 4, F_TURN_E = 8, F_BELOW = 16, F_K = 32, F_I = 64, F_SRC = 128, F_DES = 256,
       F_MON = 512, F_EDGE = 1024, F_TOP = 2048 };
constexpr uint32_t NO_PSI = 0xffffu;

// Running DFTs: fold a block of the history (steps first .. first + slots - 1)
// into the accumulators.  A brick's entries are contiguous, and 16 of an
// entry's slots are in flight at once.
struct FoldArgs {
    int items, ncd, nd, rows, nj, i0, j0, d0;
    size_t h_des, h_mon;
};

__device__ __forceinline__ void fold_dft(const StepParams &p, const FoldArgs &a, float4 *stw, int first, int slots)
{
    const int nq = p.nq, tid = threadIdx.x, NT = blockDim.x;
    const size_t plane = (size_t)p.nr * p.nphi, ndes = p.des ? plane * p.des_nk : 0;
    for (int t = tid; t < slots * nq; t += NT) {
        const float2 v = __ldg(p.t.twiddle + (size_t)first * nq + t);
        stw[t] = make_float4(v.x, v.y, -v.y, v.x);
    }
    __syncthreads();                                         // this step's history entries as well
    for (int t = tid; t < a.items; t += NT) {
        size_t entry, qs;
        float2 *out;
        if (t < 3 * a.ncd) {
            const int kk = t % a.nd, rc = t / a.nd, r = rc % a.rows, c = rc / a.rows;
            entry = a.h_des + t;
            out = p.des + c * ndes + ((size_t)(a.i0 + r / a.nj) * p.nphi + a.j0 + r % a.nj) * p.des_nk + a.d0 + kk;
            qs = 3 * ndes;
        } else {
            const int u = t - 3 * a.ncd, r = u % a.rows, c = u / a.rows;
            entry = a.h_mon + u;
            out = p.mon + c * plane + (size_t)(a.i0 + r / a.nj) * p.nphi + a.j0 + r % a.nj;
            qs = 2 * plane;
        }
        const float2 *h = p.dft_hist + entry;
        for (int l0 = 0; l0 < slots; l0 += 16) {
            float2 x[16];
#pragma unroll
            for (int l = 0; l < 16; ++l) x[l] = l0 + l < slots ? h[(size_t)(l0 + l) * p.dft_ne] : make_float2(0.f, 0.f);
            for (int w0 = 0; w0 < nq; w0 += 2) {             // n_freq is even (+-w)
                float2 *d = out + (size_t)w0 * qs;
                const float2 v0 = d[0], v1 = d[qs];
                float2 a0 = make_float2(0.f, 0.f), a1 = a0;
#pragma unroll
                for (int l = 0; l < 16; ++l) {
                    if (l0 + l < slots) {
                        const float4 u = stw[(l0 + l) * nq + w0], v = stw[(l0 + l) * nq + w0 + 1];
                        a0 = pfma(both(x[l].y), make_float2(u.z, u.w), pfma(both(x[l].x), make_float2(u.x, u.y), a0));
                        a1 = pfma(both(x[l].y), make_float2(v.z, v.w), pfma(both(x[l].x), make_float2(v.x, v.y), a1));
                    }
                }
                d[0] = padd(v0, a0);
                d[qs] = padd(v1, a1);
            }
        }
    }
}

// C own cells per thread (cell c of thread t is t + c blockDim, z fastest) and
// up to (C + 1) / 2 cells of the H layers below the brick.
template <bool RM, bool BOR, int C>
__global__ void __launch_bounds__(C == 1 ? RES_THREADS_1 : RES_THREADS, 1) k_resident(const __grid_constant__ ResidentParams q)
{
    extern __shared__ __align__(16) char sm[];
    const StepParams &p = q.p;
    const int nr = p.nr, nphi = p.nphi, nz = p.nz, nq = p.nq;
    const ResLayout L = res_layout(nr, nphi, nz, q.gi, q.gj, q.gk, BOR, RM, nq, q.nkz_h, q.nkz_e, q.nir_h, q.nir_e, q.n_recv);
    float2 *E = reinterpret_cast<float2 *>(sm + L.E), *H = reinterpret_cast<float2 *>(sm + L.H);
    float2 *pzH = reinterpret_cast<float2 *>(sm + L.pzH), *prH = reinterpret_cast<float2 *>(sm + L.prH);
    float2 *pmH = reinterpret_cast<float2 *>(sm + L.pmH), *pzE = reinterpret_cast<float2 *>(sm + L.pzE);
    float2 *prE = reinterpret_cast<float2 *>(sm + L.prE), *pmE = reinterpret_cast<float2 *>(sm + L.pmE);
    float2 *ssrc = reinterpret_cast<float2 *>(sm + L.src), *skt = reinterpret_cast<float2 *>(sm + L.kt), *sph = reinterpret_cast<float2 *>(sm + L.ph);
    float4 *stw = reinterpret_cast<float4 *>(sm + L.tw);
    uint2 *recv = reinterpret_cast<uint2 *>(sm + L.recv);
    float *itab = reinterpret_cast<float *>(sm + L.itab);
    float4 *ztab = reinterpret_cast<float4 *>(sm + L.ztab);
    int *ctl = reinterpret_cast<int *>(sm + L.ctl);

    const int tid = threadIdx.x, NT = blockDim.x;
    const int b = blockIdx.x, bk_ = b % q.gk, bj_ = (b / q.gk) % q.gj, bi_ = b / (q.gk * q.gj);
    const int i0 = brick_lo(bi_, nr, q.gi), i1 = brick_lo(bi_ + 1, nr, q.gi);
    const int j0 = brick_lo(bj_, nphi, q.gj), j1 = brick_lo(bj_ + 1, nphi, q.gj);
    const int k0 = brick_lo(bk_, nz, q.gk), k1 = brick_lo(bk_ + 1, nz, q.gk);
    const int ni = i1 - i0, nj = j1 - j0, nk = k1 - k0;
    constexpr int HJ = BOR ? 0 : 1;
    const int hi = i0 > 0 ? 1 : 0, hj = q.gj > 1 ? 1 : 0, hk = k0 > 0 ? 1 : 0;     // H layers below the brick
    const bool wrap_lo = !BOR && j0 == 0;                    // the layer below in phi is the wedge's last row
    const int NX = L.NX, SI = L.XJ * L.XK, SJ = L.XK;
    const size_t gsi = (size_t)nphi * nz, ncell = (size_t)nr * gsi;
    float2 *gE[3] = {p.f.Er, p.f.Ep, p.f.Ez}, *gH[3] = {p.f.Hr, p.f.Hp, p.f.Hz};
    const float dt = p.dt, dphi1 = BOR ? p.m : p.inv_dphi;

    // ---- fields with their halo (rows above the wedge's last times the Bloch phase; conducting walls outside)
    for (int t = tid; t < NX; t += NT) {
        const int xk = t % L.XK, xj = (t / L.XK) % L.XJ, xi = t / SI;
        const int i = i0 + xi - 1, k = k0 + xk - 1;
        int j = j0 + xj - HJ;
        float2 ph = make_float2(1.f, 0.f);
        if (!BOR && j < 0) j += nphi;
        else if (!BOR && j >= nphi) { j -= nphi; ph = p.bloch; }
        const bool in = i >= 0 && i < nr && k >= 0 && k < nz && xi <= ni + 1 && xj < nj + 2 * HJ && xk <= nk + 1;
        const size_t g = in ? (size_t)i * gsi + (size_t)j * nz + k : 0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            E[c * NX + t] = in ? turn(ph, gE[c][g]) : make_float2(0.f, 0.f);
            H[c * NX + t] = in ? gH[c][g] : make_float2(0.f, 0.f);
        }
    }
    for (int t = tid; t <= ni; t += NT) {                    // radii i0 - 1 .. i1 - 1 (row 0: the H layer below)
        const int i = max(i0 - 1 + t, 0);
        float *r = itab + t * ITAB;
        const float irn = p.t.inv_r_n[i], irh = p.t.inv_r_h[i];
        r[T_HA] = irn * dphi1; r[T_HB] = -irh * dphi1; r[T_HC] = 0.5f * irh;
        r[T_EA] = irh * dphi1; r[T_EB] = -irn * dphi1; r[T_EC] = 0.5f * irn;
        r[T_BRN] = p.t.br_n[i]; r[T_CRN] = p.t.cr_n[i];
        r[T_BRH] = p.t.br_h[i]; r[T_CRH] = p.t.cr_h[i];
        r[T_IRN] = irn; r[T_IRH] = irh;
        r[T_BMN] = p.rm.bm_n[i]; r[T_CMN] = p.rm.cm_n[i];
        r[T_BMH] = p.rm.bm_h[i]; r[T_CMH] = p.rm.cm_h[i];
    }
    for (int t = tid; t <= nk; t += NT) {                    // z positions k0 - 1 .. k1 - 1
        const int k = max(k0 - 1 + t, 0);
        ztab[t] = make_float4(p.t.bz_h[k], p.t.cz_h[k], p.t.bz_n[k], p.t.cz_n[k]);
    }
    for (int t = tid; t < nj; t += NT) {
        sph[2 * t] = p.t.ph_n[j0 + t];
        sph[2 * t + 1] = p.t.ph_h[j0 + t];
    }
    auto in_z = [&](int k) { return k < p.pz || k >= nz - p.pz; };
    auto in_r = [&](int i) { return i < p.pr_in || i >= nr - p.pr_out; };
    auto zpos = [&](int k, int from) {                       // position among the brick's PML z cells
        int n = 0;
        for (int a = from; a < k; ++a) n += in_z(a) ? 1 : 0;
        return n;
    };
    auto rpos = [&](int i, int from) {
        int n = 0;
        for (int a = from; a < i; ++a) n += in_r(a) ? 1 : 0;
        return n;
    };
    const int wH = nk + hk, njH = nj + hj, own = ni * nj * nk;
    const int pzHs = (L.ei + (q.gi > 1)) * (L.ej + (q.gj > 1)) * q.nkz_h;
    const int prHs = q.nir_h * (L.ej + (q.gj > 1)) * (L.ek + (q.gk > 1));
    const int pzEs = L.ei * L.ej * q.nkz_e, prEs = q.nir_e * L.ej * L.ek;
    const size_t gzs = 2 * (size_t)p.pz;
    auto gkz = [&](int k) { return k < p.pz ? k : k - (nz - 2 * p.pz); };
    auto gir = [&](int i) { return i < p.pr_in ? i : i - (nr - p.pr_in - p.pr_out); };
    const size_t plane = (size_t)nr * nphi, ndes = p.des ? plane * p.des_nk : 0;
    // history of the DFT sites: each brick's design cells in one piece, then each brick's monitor cells
    const int d0 = max(k0, p.des_k0) - p.des_k0, d1 = min(k1, p.des_k0 + p.des_nk) - p.des_k0;
    const int nd = p.des ? max(0, d1 - d0) : 0, ncd = ni * nj * nd, rows = ni * nj;
    const bool mon_brick = p.mon && p.mon_k >= k0 && p.mon_k < k1;
    const int dk_lo = max(p.des_k0 - k0, 0);                 // first design plane of the brick
    const size_t brick2 = (size_t)i0 * nphi + (size_t)ni * j0;
    const size_t h_des = 3 * (nd ? plane * d0 + brick2 * nd : 0), h_mon = 3 * ndes + 2 * brick2;

    // ---- this thread's cells: own ones, then cells of the layers below (H only)
    constexpr int CX = (C + 1) / 2;
    constexpr bool REG = C == 1;                             // fields in registers too (more cells would spill)
    float2 Er[C], Ep[C], Ez[C], Hr[C], Hp[C], Hz[C];
    float cr_e[C], cp_e[C], cz_e[C];                         // dt / eps of the three E sites
    uint32_t at[C], fl[C], pH[C], pE[C];                     // offset | z row << 16, flags, CPML places (z | r << 16)
    uint32_t xat[CX], xfl[CX], xpH[CX];
    // offset, flags and H-side CPML place of cell (a, jj, kk) of the brick (-1: the layer below)
    auto place = [&](int a, int jj, int kk, uint32_t &pos, uint32_t &f, uint32_t &psi) {
        const int i = i0 + a, k = k0 + kk, j = j0 + jj < 0 ? nphi - 1 : j0 + jj;
        pos = (uint32_t)(((a + 1) * L.XJ + jj + HJ) * L.XK + kk + 1) | (uint32_t)(kk + 1) << 16;
        f = F_ACT | (uint32_t)(a + 1) << 12 | (uint32_t)max(jj, 0) << 22;
        if (jj < 0 && wrap_lo) f |= F_TURN_H;                // the copy of row nphi - 1 is kept in its owner's phase
        uint32_t z = NO_PSI, r = NO_PSI;
        const size_t g2 = (size_t)i * nphi + j;
        if (in_z(k)) {
            z = ((a + hi) * njH + jj + hj) * q.nkz_h + zpos(k, k0 - hk);
            const size_t x = g2 * gzs + gkz(k);
            pzH[z] = p.psi.hr_z[x];
            pzH[pzHs + z] = p.psi.hp_z[x];
        }
        if (in_r(i)) {
            r = (rpos(i, i0 - hi) * njH + jj + hj) * wH + kk + hk;
            const size_t x = ((size_t)gir(i) * nphi + j) * nz + k;
            prH[r] = p.psi.hp_r[x];
            prH[prHs + r] = p.psi.hz_r[x];
            if (RM) {
                pmH[r] = p.rm.hr[x];
                pmH[prHs + r] = p.rm.hz[x];
            }
        }
        psi = z | r << 16;
    };
#pragma unroll
    for (int c = 0; c < C; ++c) {
        const int h = tid + c * NT;
        fl[c] = at[c] = 0;
        pH[c] = pE[c] = NO_PSI | NO_PSI << 16;
        Er[c] = Ep[c] = Ez[c] = Hr[c] = Hp[c] = Hz[c] = make_float2(0.f, 0.f);
        cr_e[c] = cp_e[c] = cz_e[c] = 0.f;
        if (h >= own) continue;
        const int kk = h % nk, jj = (h / nk) % nj, a = h / (nk * nj);
        const int i = i0 + a, j = j0 + jj, k = k0 + kk;
        uint32_t f;
        place(a, jj, kk, at[c], f, pH[c]);
        if (jj == 0 && wrap_lo) f |= F_TURN_E;
        if (jj == 0 && !hj) f |= F_BELOW;                    // the row below is this brick's own last row
        if (k > 0) f |= F_K;
        if (i > 0) f |= F_I;
        if (k == p.src_k && p.src_mode != SRC_NONE) f |= F_SRC;
        if (p.des && k >= p.des_k0 && k < p.des_k0 + p.des_nk) f |= F_DES;
        if (p.mon && k == p.mon_k) f |= F_MON;
        if ((kk == 0 && bk_ > 0) || (kk == nk - 1 && bk_ < q.gk - 1) || (a == 0 && bi_ > 0) ||
            (a == ni - 1 && bi_ < q.gi - 1) || (!BOR && q.gj > 1 && (jj == 0 || jj == nj - 1)))
            f |= F_EDGE;
        if (!BOR && q.gj == 1 && jj == 0) f |= F_TOP;        // its own row above the last
        fl[c] = f;
        const size_t g2 = (size_t)i * nphi + j, g = g2 * nz + k;
        Er[c] = gE[0][g]; Ep[c] = gE[1][g]; Ez[c] = gE[2][g];
        Hr[c] = gH[0][g]; Hp[c] = gH[1][g]; Hz[c] = gH[2][g];
        cr_e[c] = dt / (p.t.a_n[k] + p.t.d_n[k] * p.rb_r[g2]);
        cp_e[c] = dt / (p.t.a_n[k] + p.t.d_n[k] * p.rb_p[g2]);
        cz_e[c] = dt / (p.t.a_c[k] + p.t.d_c[k] * p.rb_z[g2]);
        uint32_t z = NO_PSI, r = NO_PSI;
        if (in_z(k)) {
            z = (a * nj + jj) * q.nkz_e + zpos(k, k0);
            const size_t y = g2 * gzs + gkz(k);
            pzE[z] = p.psi.er_z[y];
            pzE[pzEs + z] = p.psi.ep_z[y];
        }
        if (in_r(i)) {
            r = (rpos(i, i0) * nj + jj) * nk + kk;
            const size_t x = ((size_t)gir(i) * nphi + j) * nz + k;
            prE[r] = p.psi.ep_r[x];
            prE[prEs + r] = p.psi.ez_r[x];
            if (RM) {
                pmE[r] = p.rm.er[x];
                pmE[prEs + r] = p.rm.ez[x];
            }
        }
        pE[c] = z | r << 16;
    }
    const int lay_i = hi * njH * wH, lay_j = hj * ni * wH, lay_k = hk * ni * nj;
#pragma unroll
    for (int c = 0; c < CX; ++c) {
        int h = tid + c * NT;
        xfl[c] = xat[c] = 0;
        xpH[c] = NO_PSI | NO_PSI << 16;
        if (h >= lay_i + lay_j + lay_k) continue;
        int a = -1, jj, kk;
        if (h < lay_i) {
            kk = h % wH - hk;
            jj = h / wH - hj;
        } else if (h -= lay_i; h < lay_j) {
            kk = h % wH - hk;
            jj = -1;
            a = h / wH;
        } else {
            h -= lay_j;
            kk = -1;
            jj = h % nj;
            a = h / nj;
        }
        place(a, jj, kk, xat[c], xfl[c], xpH[c]);
    }
    // ---- halo list: the packet of each halo value of E and its place
    if (tid == 0) ctl[0] = 0;
    __syncthreads();
    for (int t = tid; t < NX; t += NT) {
        const int xk = t % L.XK, xj = (t / L.XK) % L.XJ, xi = t / SI;
        if (xi > ni + 1 || xj >= nj + 2 * HJ || xk > nk + 1) continue;
        const int di = xi == 0 ? -1 : (xi == ni + 1 ? 1 : 0), dk = xk == 0 ? -1 : (xk == nk + 1 ? 1 : 0);
        const int dj = BOR ? 0 : (xj == 0 ? -1 : (xj == nj + 1 ? 1 : 0));
        const int need = halo_need(di, dj, dk);
        const int i = i0 + xi - 1, k = k0 + xk - 1;
        int j = j0 + xj - HJ, wrap = 0;
        if (!need || i < 0 || i >= nr || k < 0 || k >= nz) continue;
        if (!BOR && j < 0) j += nphi;
        else if (!BOR && j >= nphi) { j -= nphi; wrap = 1; }
        if (q.gj == 1 && (dj < 0 || (dj > 0 && di == 0 && dk == 0))) continue;     // own rows: no copy below, F_TOP above
        for (int c = 0; c < 3; ++c) {
            if (!(need >> c & 1)) continue;
            const int e = atomicAdd(ctl, 1);
            if (e < q.n_recv)
                recv[e] = make_uint2((uint32_t)((size_t)c * ncell + (size_t)i * gsi + (size_t)j * nz + k),
                                     (uint32_t)(c * NX + t) | (uint32_t)wrap << 30);
        }
    }
    __syncthreads();
    const int nrecv = min(ctl[0], q.n_recv);

    // Source of a step, by step parity: the pulse, or per radius sum_q beta_q(r) k_q(t) of an adjoint run.  The
    // time table comes in blocks of SRC_BLOCK steps, a step ahead: loaded when needed, its latency was 1000-2000
    // cycles of every step.
    const bool src_brick = p.src_mode != SRC_NONE && p.src_k >= k0 && p.src_k < k1;
    const bool adjoint = p.src_mode == SRC_ADJOINT;
    auto fill_times = [&](int first) {                       // steps first .. first + SRC_BLOCK - 1, a multiple of it
        if (!src_brick) return;
        const int w = adjoint ? nq : 1, m = min(SRC_BLOCK, q.n_steps - first) * w;
        float2 *d = skt + (first / SRC_BLOCK & 1) * SRC_BLOCK * nq;
        for (int t = tid; t < m; t += NT)
            d[t] = adjoint ? p.t.adj_time[(size_t)first * nq + t] : both(p.t.pulse[first + t] * p.src_scale);
    };
    auto fill_source = [&](int n) {
        if (!src_brick) return;
        float2 *s = ssrc + (n & 1) * 2 * (L.ei + 1);
        const float2 *kt = skt + (n / SRC_BLOCK & 1) * SRC_BLOCK * nq + (n % SRC_BLOCK) * (adjoint ? nq : 1);
        if (!adjoint) {
            if (tid == 0) s[0] = kt[0];
            return;
        }
        for (int t = tid; t < 2 * ni; t += NT) {
            const int c = t >= ni ? 1 : 0, i = c ? t - ni : t;
            const float2 *bt = c ? p.beta_p : p.beta_r;
            float2 v = make_float2(0.f, 0.f);
            for (int w = 0; w < nq; ++w) v = c_fma(__ldg(bt + (size_t)w * nr + i0 + i), kt[w], v);
            s[c * (L.ei + 1) + i] = v;
        }
    };
    fill_times(q.n0);
    __syncthreads();
    fill_source(q.n0);
    FoldArgs fa{};
    fa.items = p.des || p.mon ? 3 * ncd + (mon_brick ? 2 * rows : 0) : 0;
    fa.ncd = ncd; fa.nd = nd; fa.rows = rows; fa.nj = nj; fa.i0 = i0; fa.j0 = j0; fa.d0 = d0;
    fa.h_des = h_des; fa.h_mon = h_mon;
    const float2 c_dz = both(p.inv_dz), c_ndz = both(-p.inv_dz), c_dr = both(p.inv_dr);
    const float2 c_dt = both(dt), c_ndt = both(-dt);
    const float2 *E1 = E + NX, *E2 = E + 2 * NX, *H1 = H + NX, *H2 = H + 2 * NX;
    __syncthreads();

    // H^{n+1/2} of one cell from E around it
    auto update_h = [&](uint32_t f, uint32_t pos, uint32_t psi, float2 er, float2 ep, float2 ez, float2 &hr, float2 &hp,
                        float2 &hz) {
        const int o = pos & 0xffffu;
        const float *it = itab + (f >> 12 & 1023u) * ITAB;
        float2 gz, gr;                                       // phi differences of E_z, E_r (i F on the axis zone)
        if (BOR) {
            gz = make_float2(-ez.y, ez.x);
            gr = make_float2(-er.y, er.x);
        } else {
            float2 ez_j = E2[o + SJ], er_j = E[o + SJ];
            if (f & F_TURN_H) {
                ez_j = turn(p.bloch, ez_j);
                er_j = turn(p.bloch, er_j);
            }
            gz = psub(ez_j, ez);
            gr = psub(er_j, er);
        }
        const float2 ep_i = E1[o + SI];
        const float2 dzp = psub(E1[o + 1], ep), dzr = psub(E[o + 1], er), drz = psub(E2[o + SI], ez);
        const float2 df = psub(ep_i, ep), sf = padd(ep_i, ep);
        float2 tr = pmul(dzp, c_ndz);                        // curls of H_r, of H_phi, of H_z; dt joins them in the last fma
        float2 tp = pfma(dzr, c_ndz, pmul(drz, c_dr));
        float2 tz = pfma(sf, both(it[T_HC]), pmul(df, c_dr));
        const uint32_t pz = psi & 0xffffu, pr = psi >> 16;
        if (pz != NO_PSI) {
            const float4 zt = ztab[pos >> 16];
            const float2 bz = both(zt.x), cz = both(zt.y);
            const float2 u = pfma(pzH[pz], bz, pmul(pmul(dzp, c_dz), cz));
            const float2 v = pfma(pzH[pzHs + pz], bz, pmul(pmul(dzr, c_dz), cz));
            pzH[pz] = u;
            pzH[pzHs + pz] = v;
            tr = psub(tr, u);
            tp = psub(tp, v);
        }
        if (pr != NO_PSI) {
            const float2 br = both(it[T_BRH]), cr = both(it[T_CRH]);
            const float2 u = pfma(prH[pr], br, pmul(pmul(drz, c_dr), cr));
            prH[pr] = u;
            tp = padd(tp, u);
            if (RM) {                                        // only the derivative is stretched; the rest over r~
                const float2 d = pmul(df, c_dr);
                const float2 w = pfma(prH[prHs + pr], br, pmul(d, cr));
                prH[prHs + pr] = w;
                const float2 X = pmul(gz, both(dphi1));
                const float2 m = pfma(pmH[pr], both(it[T_BMN]), pmul(X, both(it[T_CMN])));
                pmH[pr] = m;
                tr = pfma(padd(X, m), both(it[T_IRN]), tr);
                const float2 Y = pfma(sf, both(0.5f), pmul(gr, both(-dphi1)));
                const float2 mz = pfma(pmH[prHs + pr], both(it[T_BMH]), pmul(Y, both(it[T_CMH])));
                pmH[prHs + pr] = mz;
                tz = pfma(padd(Y, mz), both(it[T_IRH]), padd(d, w));
            } else {
                const float2 w = pfma(prH[prHs + pr], br, pmul(tz, cr));
                prH[prHs + pr] = w;
                tz = padd(tz, w);
            }
        }
        if (!RM || pr == NO_PSI) {
            tr = pfma(gz, both(it[T_HA]), tr);
            tz = pfma(gr, both(it[T_HB]), tz);
        }
        H[o] = hr = pfma(tr, c_ndt, hr);
        H[NX + o] = hp = pfma(tp, c_dt, hp);
        H[2 * NX + o] = hz = pfma(tz, c_ndt, hz);
    };

    for (int n = q.n0; n < q.n1; ++n) {
        // the cells' addresses are worked out anew in each step: kept over the loop they would spill
#pragma unroll
        for (int c = 0; c < C; ++c) asm volatile("" : "+r"(at[c]), "+r"(fl[c]), "+r"(pH[c]), "+r"(pE[c]));
#pragma unroll
        for (int c = 0; c < CX; ++c) asm volatile("" : "+r"(xat[c]), "+r"(xfl[c]), "+r"(xpH[c]));
        // ---- H^{n+1/2} of the brick and of the layers below it
#pragma unroll
        for (int c = 0; c < C; ++c) {
            if (!fl[c]) continue;
            const int o = at[c] & 0xffffu;
            if (!REG) {
                Er[c] = E[o]; Ep[c] = E1[o]; Ez[c] = E2[o];
                Hr[c] = H[o]; Hp[c] = H1[o]; Hz[c] = H2[o];
            }
            update_h(fl[c], at[c], pH[c], Er[c], Ep[c], Ez[c], Hr[c], Hp[c], Hz[c]);
        }
#pragma unroll
        for (int c = 0; c < CX; ++c) {
            if (!xfl[c]) continue;
            const int o = xat[c] & 0xffffu;
            float2 hr = H[o], hp = H1[o], hz = H2[o];
            update_h(xfl[c], xat[c], xpH[c], E[o], E1[o], E2[o], hr, hp, hz);
        }
        __syncthreads();

        // ---- E^{n+1} of the brick
#pragma unroll
        for (int c = 0; c < C; ++c) asm volatile("" : "+r"(at[c]), "+r"(fl[c]), "+r"(pE[c]));
        const uint32_t tag = (uint32_t)(n + 1);
        uint4 *box = q.mail + (size_t)(n & 1) * 3 * ncell;
        float2 *hs = p.dft_hist + (size_t)(n % DFT_BLOCK) * p.dft_ne;
        const float2 *src = ssrc + (n & 1) * 2 * (L.ei + 1);
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const uint32_t f = fl[c];
            if (!f) continue;
            const int o = at[c] & 0xffffu;
            const float *it = itab + (f >> 12 & 1023u) * ITAB;
            float2 hr = Hr[c], hp = Hp[c], hz = Hz[c];
            if (!REG) { hr = H[o]; hp = H1[o]; hz = H2[o]; }
            float2 gz, gr;                                   // phi differences of H_z, H_r
            if (BOR) {
                gz = make_float2(-hz.y, hz.x);
                gr = make_float2(-hr.y, hr.x);
            } else {
                const int below = f & F_BELOW ? o + (nj - 1) * SJ : o - SJ;
                float2 hz_j = H2[below], hr_j = H[below];
                if (f & F_TURN_E) {
                    hz_j = turn(p.bloch_inv, hz_j);
                    hr_j = turn(p.bloch_inv, hr_j);
                }
                gz = psub(hz, hz_j);
                gr = psub(hr, hr_j);
            }
            const float2 hp_i = H1[o - SI];
            const float2 dzp = psub(hp, H1[o - 1]), dzr = psub(hr, H[o - 1]), drz = psub(hz, H2[o - SI]);
            const float2 df = psub(hp, hp_i), sf = padd(hp, hp_i);
            float2 tr = pmul(dzp, c_ndz);
            float2 tp = pfma(dzr, c_dz, pmul(drz, both(-p.inv_dr)));
            float2 tz = pfma(sf, both(it[T_EC]), pmul(df, c_dr));
            const uint32_t pz = pE[c] & 0xffffu, pr = pE[c] >> 16;
            if (pz != NO_PSI && (f & F_K)) {
                const float4 zt = ztab[at[c] >> 16];
                const float2 bz = both(zt.z), cz = both(zt.w);
                const float2 u = pfma(pzE[pz], bz, pmul(pmul(dzp, c_dz), cz));
                pzE[pz] = u;
                tr = psub(tr, u);
                if (f & F_I) {
                    const float2 v = pfma(pzE[pzEs + pz], bz, pmul(pmul(dzr, c_dz), cz));
                    pzE[pzEs + pz] = v;
                    tp = padd(tp, v);
                }
            }
            if (pr != NO_PSI) {
                const float2 br = both(it[T_BRN]), cr = both(it[T_CRN]);
                if ((f & (F_I | F_K)) == (F_I | F_K)) {
                    const float2 u = pfma(prE[pr], br, pmul(pmul(drz, c_dr), cr));
                    prE[pr] = u;
                    tp = psub(tp, u);
                }
                if (RM) {
                    if (f & F_K) {
                        const float2 X = pmul(gz, both(dphi1));
                        const float2 m = pfma(pmE[pr], both(it[T_BMH]), pmul(X, both(it[T_CMH])));
                        pmE[pr] = m;
                        tr = pfma(padd(X, m), both(it[T_IRH]), tr);
                    }
                    if (f & F_I) {
                        const float2 d = pmul(df, c_dr);
                        const float2 w = pfma(prE[prEs + pr], br, pmul(d, cr));
                        prE[prEs + pr] = w;
                        const float2 Y = pfma(sf, both(0.5f), pmul(gr, both(-dphi1)));
                        const float2 mz = pfma(pmE[prEs + pr], both(it[T_BMN]), pmul(Y, both(it[T_CMN])));
                        pmE[prEs + pr] = mz;
                        tz = pfma(padd(Y, mz), both(it[T_IRN]), padd(d, w));
                    }
                } else if (f & F_I) {
                    const float2 w = pfma(prE[prEs + pr], br, pmul(tz, cr));
                    prE[prEs + pr] = w;
                    tz = padd(tz, w);
                }
            }
            if (!RM || pr == NO_PSI) {
                tr = pfma(gz, both(it[T_EA]), tr);
                tz = pfma(gr, both(it[T_EB]), tz);
            }
            if (f & F_SRC) {
                const int a = (int)(f >> 12 & 1023u) - 1;
                const float2 pn = sph[2 * (f >> 22)], ph = sph[2 * (f >> 22) + 1];
                float2 jr, jp;
                if (p.src_mode == SRC_PLANE_WAVE) {          // m = +1 part of an x-polarised sheet
                    const float s = src[0].x;
                    jr = c_scale(pn, s);
                    jp = make_float2(-ph.y * s, ph.x * s);
                } else {
                    jr = c_mul(pn, src[a]);
                    jp = c_mul(ph, src[L.ei + 1 + a]);
                }
                tr = psub(tr, jr);
                tp = psub(tp, jp);
            }
            // conducting walls: E_r, E_phi vanish at k = 0, E_phi, E_z at i = 0
            float2 er = Er[c], ep = Ep[c], ez = Ez[c];
            if (!REG) { er = E[o]; ep = E1[o]; ez = E2[o]; }
            if (f & F_K) er = pfma(tr, both(cr_e[c]), er);
            if ((f & (F_I | F_K)) == (F_I | F_K)) ep = pfma(tp, both(cp_e[c]), ep);
            if (f & F_I) ez = pfma(tz, both(cz_e[c]), ez);
            const int a = (int)(f >> 12 & 1023u) - 1, jj = f >> 22, kk = (int)(at[c] >> 16) - 1;
            if (f & F_EDGE) {
                uint4 *m = box + (uint32_t)(((i0 + a) * nphi + j0 + jj) * nz + k0 + kk);
                send_packet(m, er, tag);
                send_packet(m + ncell, ep, tag);
                send_packet(m + 2 * ncell, ez, tag);
            }
            E[o] = er;
            E[NX + o] = ep;
            E[2 * NX + o] = ez;
            if (REG) { Er[c] = er; Ep[c] = ep; Ez[c] = ez; }
            if (f & F_TOP) {
                E[o + nj * SJ] = turn(p.bloch, er);
                E[2 * NX + o + nj * SJ] = turn(p.bloch, ez);
            }
            if (f & F_DES) {
                float2 *d = hs + h_des + ((a * nj + jj) * nd + kk - dk_lo);
                d[0] = er;
                d[ncd] = ep;
                d[2 * ncd] = ez;
            }
            if (f & F_MON) {
                float2 *d = hs + h_mon + a * nj + jj;
                d[0] = er;
                d[rows] = ep;
            }
        }

        // ---- running DFTs, while the neighbours' packets are under way
        if (fa.items && (n % DFT_BLOCK == DFT_BLOCK - 1 || n + 1 == q.n_steps))
            fold_dft(p, fa, stw, n - n % DFT_BLOCK, n % DFT_BLOCK + 1);
        if (n + 1 == q.n1) break;

        // ---- halo of E^{n+1}
        fill_source(n + 1);
        if (n % SRC_BLOCK == SRC_BLOCK - 2 && n + 2 < q.n_steps) fill_times(n + 2);
        bool bad = false;
        {
            const uint32_t want = q.inject_timeout ? 0xffffffffu : tag;
            int polls = 0;
            u64 since = 0;
            for (int e0 = tid; e0 < nrecv && !bad; e0 += 4 * NT) {
                uint2 r[4];
                int open = 0;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (e0 + u * NT < nrecv) {
                        r[u] = recv[e0 + u * NT];
                        open |= 1 << u;
                    }
                while (open) {
                    u64 lo[4], hi[4];                        // all loads of a round in flight before the first is looked at
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (open >> u & 1) read_packet(box + r[u].x, lo[u], hi[u]);
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if ((open >> u & 1) && (uint32_t)(lo[u] >> 32) == want && (uint32_t)(hi[u] >> 32) == want) {
                            const float2 v = make_float2(__uint_as_float((uint32_t)lo[u]), __uint_as_float((uint32_t)hi[u]));
                            E[r[u].y & 0x3fffffffu] = r[u].y >> 30 ? turn(p.bloch, v) : v;
                            open &= ~(1 << u);
                        }
                    if (!open) break;
                    bad = ++polls >= q.wait_limit;           // bounded: the polls, two seconds, or another brick gave up
                    if ((polls & 63) == 0) {
                        const u64 t = now_ns();
                        if (!since) since = t;
                        bad = bad || t - since > 2000000000ull || *(volatile int *)q.err;
                    }
                    if (bad) break;
                }
            }
        }
        if (bad) atomicExch(q.err, 1);
        if (__syncthreads_or(bad)) return;
    }

    // ---- state back to the field arrays (each thread its own cells: nothing to wait for)
#pragma unroll
    for (int c = 0; c < C; ++c) {
        if (!fl[c]) continue;
        const int k = k0 - 1 + (int)(at[c] >> 16), i = i0 + (int)(fl[c] >> 12 & 1023u) - 1;
        const size_t g2 = (size_t)i * nphi + j0 + (fl[c] >> 22), g = g2 * nz + k;
        const int o = at[c] & 0xffffu;
#pragma unroll
        for (int w = 0; w < 3; ++w) {
            gE[w][g] = E[w * NX + o];
            gH[w][g] = H[w * NX + o];
        }
        const uint32_t zh = pH[c] & 0xffffu, rh = pH[c] >> 16, ze = pE[c] & 0xffffu, re = pE[c] >> 16;
        if (zh != NO_PSI) {
            const size_t x = g2 * gzs + gkz(k);
            p.psi.hr_z[x] = pzH[zh];
            p.psi.hp_z[x] = pzH[pzHs + zh];
            p.psi.er_z[x] = pzE[ze];
            p.psi.ep_z[x] = pzE[pzEs + ze];
        }
        if (rh != NO_PSI) {
            const size_t x = ((size_t)gir(i) * nphi + (g2 - (size_t)i * nphi)) * nz + k;
            p.psi.hp_r[x] = prH[rh];
            p.psi.hz_r[x] = prH[prHs + rh];
            p.psi.ep_r[x] = prE[re];
            p.psi.ez_r[x] = prE[prEs + re];
            if (RM) {
                p.rm.hr[x] = pmH[rh];
                p.rm.hz[x] = pmH[prHs + rh];
                p.rm.er[x] = pmE[re];
                p.rm.ez[x] = pmE[prEs + re];
            }
        }
    }
}

typedef void (*ResKernel)(const ResidentParams);

template <int C>
ResKernel res_kernel_c(const StepParams &p)
{
    if (p.bor) return p.rpml_metric ? k_resident<true, true, C> : k_resident<false, true, C>;
    return p.rpml_metric ? k_resident<true, false, C> : k_resident<false, false, C>;
}

ResKernel res_kernel(const StepParams &p, int per_thread)
{
    switch (per_thread) {
    case 1: return res_kernel_c<1>(p);
    case 2: return res_kernel_c<2>(p);
    case 3: return res_kernel_c<3>(p);
    default: return res_kernel_c<4>(p);
    }
}

// Slab extents and halo entries of the largest brick of a cut.
struct ResExtents { int nkz_h = 0, nkz_e = 0, nir_h = 0, nir_e = 0, n_recv = 0; };

ResExtents res_extents(const StepParams &p, int gi, int gj, int gk)
{
    ResExtents x;
    auto slabs = [](int lo, int hi, int in, int out_from) {
        int n = 0;
        for (int a = lo; a < hi; ++a) n += (a < in || a >= out_from) ? 1 : 0;
        return n;
    };
    for (int b = 0; b < gk; ++b) {
        const int lo = brick_lo(b, p.nz, gk), hi = brick_lo(b + 1, p.nz, gk);
        x.nkz_e = std::max(x.nkz_e, slabs(lo, hi, p.pz, p.nz - p.pz));
        x.nkz_h = std::max(x.nkz_h, slabs(std::max(lo - 1, 0), hi, p.pz, p.nz - p.pz));
    }
    for (int b = 0; b < gi; ++b) {
        const int lo = brick_lo(b, p.nr, gi), hi = brick_lo(b + 1, p.nr, gi);
        x.nir_e = std::max(x.nir_e, slabs(lo, hi, p.pr_in, p.nr - p.pr_out));
        x.nir_h = std::max(x.nir_h, slabs(std::max(lo - 1, 0), hi, p.pr_in, p.nr - p.pr_out));
    }
    const int ei = (p.nr + gi - 1) / gi, ej = (p.nphi + gj - 1) / gj, ek = (p.nz + gk - 1) / gk;
    for (int di = -1; di <= 1; ++di)
        for (int dj = -1; dj <= 1; ++dj)
            for (int dk = -1; dk <= 1; ++dk) {
                if ((di && gi == 1) || (dk && gk == 1) || (dj && (p.bor || (gj == 1 && (dj < 0 || (!di && !dk)))))) continue;
                const int need = halo_need(di, dj, dk);
                const int n = (need & 1) + (need >> 1 & 1) + (need >> 2 & 1);
                x.n_recv += n * (di ? 1 : ei) * (dj ? 1 : ej) * (dk ? 1 : ek);
            }
    x.n_recv = std::max(x.n_recv, 1);
    return x;
}

}  // namespace

size_t resident_mail_bytes(int nr, int nphi, int nz) { return (size_t)2 * 3 * nr * nphi * nz * sizeof(uint4); }

ResidentPlan resident_plan(const StepParams &p, int sms, size_t smem_limit)
{
    ResidentPlan best;
    double best_cost = 1e30;
    const long long cells = (long long)p.nr * p.nphi * p.nz;
    const long long most = (long long)RES_THREADS * RES_MAX_CELLS;
    if (cells > most * sms || p.nr > 1000 || p.nphi > 1000) return best;
    for (int gi = 1; gi <= std::min(sms, p.nr); ++gi)
        for (int gj = 1; gi * gj <= sms && gj <= p.nphi; ++gj)
            for (int gk = 1; gi * gj * gk <= sms && gk <= p.nz; ++gk) {
                const int ei = (p.nr + gi - 1) / gi, ej = (p.nphi + gj - 1) / gj, ek = (p.nz + gk - 1) / gk;
                const long long h = (long long)(ei + (gi > 1)) * (ej + (gj > 1)) * (ek + (gk > 1));
                const long long own = (long long)ei * ej * ek;
                if (own > most) continue;
                const int per = own <= RES_THREADS_1 ? 1 : std::max(2, (int)((own + RES_THREADS - 1) / RES_THREADS));
                const int threads = (int)(((own + per - 1) / per + 31) / 32 * 32);
                if (h - own > (long long)threads * ((per + 1) / 2)) continue;
                const int faces = 5 * ((gi > 1) * ej * ek + (gj > 1) * ei * ek + (gk > 1) * ei * ej);
                // 8-byte shared-memory accesses go by half warps: rows of 16 cells keep them off the same banks
                const double rows = ek % 16 == 0 ? 1.0 : (ek >= 24 ? 1.2 : 1.4);
                const double cost = (double)h * rows + 0.3 * faces + 0.05 * gi * gj * gk;
                if (cost >= best_cost) continue;
                const ResExtents x = res_extents(p, gi, gj, gk);
                const ResLayout L = res_layout(p.nr, p.nphi, p.nz, gi, gj, gk, p.bor, p.rpml_metric, p.nq, x.nkz_h, x.nkz_e,
                                               x.nir_h, x.nir_e, x.n_recv);
                if (L.NX > 0xffff || (size_t)L.bytes > smem_limit) continue;
                best_cost = cost;
                best.gi = gi; best.gj = gj; best.gk = gk;
                best.per_thread = per;
                best.threads = std::max(threads, std::min(per == 1 ? RES_THREADS_1 : RES_THREADS, (x.n_recv + 31) / 32 * 32));   // a thread per packet
                best.smem = (size_t)L.bytes;
            }
    return best;
}

cudaError_t launch_resident(const ResidentPlan &pl, const StepParams &p, int n0, int n1, int n_steps, void *mail,
                            int *err, int wait_limit, int inject_timeout, cudaStream_t s)
{
    const ResExtents x = res_extents(p, pl.gi, pl.gj, pl.gk);
    ResidentParams q{};
    q.p = p;
    q.gi = pl.gi; q.gj = pl.gj; q.gk = pl.gk;
    q.nkz_h = x.nkz_h; q.nkz_e = x.nkz_e; q.nir_h = x.nir_h; q.nir_e = x.nir_e;
    q.n_recv = x.n_recv;
    q.n0 = n0; q.n1 = n1; q.n_steps = n_steps;
    q.mail = (uint4 *)mail;
    q.err = err;
    q.wait_limit = wait_limit;
    q.inject_timeout = inject_timeout;
    ResKernel k = res_kernel(p, pl.per_thread);
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pl.smem);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(pl.blocks());
    cfg.blockDim = dim3(pl.threads);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, q);
}

}  // namespace zda
